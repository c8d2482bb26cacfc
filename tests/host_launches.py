"""What the library asks the CUDA runtime for, without a device: the calls run in a child process against a stand-in
runtime that writes every launch, event and copy down and launches nothing. Addresses are never followed."""
from __future__ import annotations

import os
import shutil
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

RUNTIME = r"""
#include <cuda.h>
#include <cuda_runtime_api.h>
#include <stdio.h>
#include <string.h>
static struct { const void* host; const char* name; } known[256];
static int n_known;
static char handle[16][8];
void** __cudaRegisterFatBinary(void* f) { (void)f; return (void**)handle[0]; }
void __cudaRegisterFatBinaryEnd(void** h) { (void)h; }
void __cudaUnregisterFatBinary(void** h) { (void)h; }
void __cudaRegisterVar(void** h, char* a, char* b, const char* c, int e, size_t s, int k, int g) {
  (void)h; (void)a; (void)b; (void)c; (void)e; (void)s; (void)k; (void)g;
}
void __cudaRegisterFunction(void** h, const char* host, char* dev, const char* name, int lim, uint3* t, uint3* b, dim3* bd,
                            dim3* gd, int* w) {
  (void)h; (void)dev; (void)lim; (void)t; (void)b; (void)bd; (void)gd; (void)w;
  if (n_known < 256) { known[n_known].host = host; known[n_known++].name = name; }
}
static CUresult encode(CUtensorMap* m, CUtensorMapDataType a, cuuint32_t r, void* p, const cuuint64_t* d, const cuuint64_t* s,
                       const cuuint32_t* b, const cuuint32_t* e, CUtensorMapInterleave i, CUtensorMapSwizzle w,
                       CUtensorMapL2promotion l, CUtensorMapFloatOOBfill f) {
  (void)a; (void)r; (void)p; (void)d; (void)s; (void)b; (void)e; (void)i; (void)w; (void)l; (void)f;
  memset(m, 0, sizeof(*m));
  return CUDA_SUCCESS;
}
cudaError_t cudaGetDriverEntryPoint(const char* s, void** fn, unsigned long long f, enum cudaDriverEntryPointQueryResult* q) {
  (void)s; (void)f;
  *fn = (void*)encode;
  if (q) *q = cudaDriverEntryPointSuccess;
  return cudaSuccess;
}
cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaSetDevice(int d) { (void)d; return cudaSuccess; }
cudaError_t cudaGetLastError(void) { return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, enum cudaDeviceAttr a, int d) { (void)a; (void)d; *v = 148; return cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void* f, enum cudaFuncAttribute a, int v) { (void)f; (void)a; (void)v; return cudaSuccess; }
cudaError_t cudaGetSymbolAddress(void** p, const void* s) { (void)s; *p = (void*)(1ull << 36); return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned f) { static int n; (void)f; *s = (cudaStream_t)(size_t)(900 + n++); return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t s) { (void)s; return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned f) { static int n; (void)f; *e = (cudaEvent_t)(size_t)(700 + n++); return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t e) { (void)e; return cudaSuccess; }
cudaError_t cudaStreamQuery(cudaStream_t s) { (void)s; return cudaSuccess; }
cudaError_t cudaThreadExchangeStreamCaptureMode(enum cudaStreamCaptureMode* m) { (void)m; return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t s, enum cudaStreamCaptureStatus* st) { (void)s; *st = cudaStreamCaptureStatusNone; return cudaSuccess; }
cudaError_t cudaStreamGetCaptureInfo_v2(cudaStream_t s, enum cudaStreamCaptureStatus* st, unsigned long long* id, cudaGraph_t* g,
                                        const cudaGraphNode_t** d, size_t* n) {
  (void)s; (void)id; (void)g; (void)d; (void)n;
  *st = cudaStreamCaptureStatusNone;
  return cudaSuccess;
}
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) { printf("record %zu %zu\n", (size_t)s, (size_t)e); return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned f) { (void)f; printf("wait %zu %zu\n", (size_t)s, (size_t)e); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, enum cudaMemcpyKind k, cudaStream_t st) {
  (void)d; (void)s; (void)k;
  printf("copy %zu %zu\n", (size_t)st, n);
  return cudaSuccess;
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void** args) {
  const char* name = "?";
  unsigned dependent = 0, cluster = 1;
  (void)args;
  for (int i = 0; i < n_known; ++i) if (known[i].host == f) name = known[i].name;
  for (unsigned i = 0; i < c->numAttrs; ++i) {
    if (c->attrs[i].id == cudaLaunchAttributeProgrammaticStreamSerialization) dependent = c->attrs[i].val.programmaticStreamSerializationAllowed;
    if (c->attrs[i].id == cudaLaunchAttributeClusterDimension) cluster = c->attrs[i].val.clusterDim.x;
  }
  printf("launch %zu %s %u %u %u\n", (size_t)c->stream, name, c->gridDim.x, cluster, dependent);
  return cudaSuccess;
}
"""

CHILD = """
import ctypes, sys
from unittest import mock
sys.modules["torch"] = mock.MagicMock()           # (torch would bring the real runtime)
sys.path.insert(0, {root!r})
ctypes.CDLL({lib!r}, ctypes.RTLD_GLOBAL)
libc = ctypes.CDLL(None)
from paper_2601_23180_b200 import binding as ts
from tests.test_fused_arguments import Args
lib, r = ts._lib, ctypes.byref
def call(name, rc):
    libc.fflush(None)
    print("call", name, rc, flush=True)
{code}
"""


class Launch:
    def __init__(self, stream, kernel, grid, cluster, dependent):
        self.stream, self.kernel, self.grid, self.cluster, self.dependent = int(stream), kernel, int(grid), int(cluster), int(dependent)


def requests(tmp_path, code):
    """Runs `code` (it has ts, lib, r = byref, Args and call(name, status), which ends a call of the library) against
    the stand-in. {name: [(what, stream, event, bytes or Launch)]}"""
    cc = shutil.which("gcc") or shutil.which("cc")
    cuda = next((d for d in (os.environ.get("CUDA_HOME"), "/usr/local/cuda") if d and os.path.exists(d + "/include/cuda.h")), None)
    if not cc or not cuda:
        pytest.skip("no C compiler or CUDA headers")
    src, so = tmp_path / "runtime.c", tmp_path / "runtime.so"
    src.write_text(RUNTIME)
    subprocess.run([cc, "-shared", "-fPIC", "-O1", "-I", cuda + "/include", "-o", str(so), str(src)], check=True)
    out = subprocess.run([sys.executable, "-c", CHILD.format(root=ROOT, lib=str(so), code=code)], capture_output=True, text=True,
                         cwd=ROOT, timeout=300)
    assert out.returncode == 0, out.stderr[-3000:]
    calls, now = {}, []
    for line in out.stdout.splitlines():
        what, *rest = line.split()
        if what == "call":
            assert rest[1] == "0", line
            calls[rest[0]], now = now, []
        elif what == "launch":
            now.append((what, int(rest[0]), Launch(*rest)))
        else:
            now.append((what, int(rest[0]), int(rest[1])))
    return calls
