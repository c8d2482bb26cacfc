"""The fused pass of few rows, whose attention runs beside the LM head in one CTA per (sequence, KV head, M tile)
that takes the splits of the attention's own plan in turn: the same bits as the attention called by itself."""
import math

import pytest

pytestmark = pytest.mark.gpu


class Pass:
    """One pass with inputs drawn on the GPU. Capacity `cap` tokens per sequence, lengths `lens`."""

    def __init__(self, T, Hq, Hkv, cap, lens, listed=None, n_nodes=None, paged=False, d=2048, V=151936, seed=3, target=False):
        import torch
        from paper_2601_23180_b200 import binding as ts
        B = len(lens)
        g = torch.Generator(device="cuda")
        g.manual_seed(seed)

        def normal(*shape):
            return torch.randn(*shape, generator=g, device="cuda", dtype=torch.bfloat16)

        def i32(x):
            return torch.tensor(x, dtype=torch.int32, device="cuda")

        self.B, self.T, self.scale = B, T, 1.0 / math.sqrt(128)
        self.q, self.kt, self.vt = normal(B, T, Hq, 128), normal(B, T, Hkv, 128), normal(B, T, Hkv, 128)
        self.table = None
        if paged:
            blocks = (cap + 63) // 64
            self.table = torch.randperm(B * blocks, generator=g, device="cuda").to(torch.int32).view(B, blocks).contiguous()
            self.kc, self.vc = normal(B * blocks, 64, Hkv, 128), normal(B * blocks, 64, Hkv, 128)
        else:
            self.kc, self.vc = normal(B, cap, Hkv, 128), normal(B, cap, Hkv, 128)
        self.ctx, self.lens = i32(lens), lens
        self.parent = i32([[-1] + [(7 * i + 3 * b) % i for i in range(1, T)] for b in range(B)])
        self.tok = torch.randint(0, V, (B, T), generator=g, device="cuda", dtype=torch.int32)
        self.W, self.h = normal(V, d).mul_(0.02), normal(B, T, d)
        self.seqs = list(range(B)) if listed is None else listed
        self.index = None if listed is None else i32(listed)
        self.nodes = None if n_nodes is None else i32(n_nodes)
        self.n_nodes = n_nodes or [T] * B
        self.status = torch.zeros(1, dtype=torch.int32, device="cuda")
        self.mask = torch.zeros((B, T), dtype=torch.int64, device="cuda")
        self.depth = torch.zeros((B, T), dtype=torch.int32, device="cuda")
        self.o = torch.zeros((B, T, Hq, 128), dtype=torch.bfloat16, device="cuda")
        self.lse = torch.zeros((B, Hq, T), dtype=torch.float32, device="cuda")
        self.stats, self.out = ts.alloc_stats(B, T), ts.alloc_scan_out(B, T)
        self.tree_args = ts.tree_args(self.parent, self.mask, self.depth, dev_status=self.status)
        self.attn_args = ts.attn_args(self.q, self.kt, self.vt, self.mask, self.kc, self.vc, self.ctx, self.scale, self.o,
                                      block_table=self.table, seq_index=self.index, lse=self.lse, dev_status=self.status,
                                      n_nodes=self.nodes)
        self.ws = []
        self.lm_args = ts.lmhead_args(self.h, self.W, self.parent, self.tok, 2.0, self.stats, seq_index=self.index,
                                      dev_status=self.status)
        for a, need in ((self.attn_args, ts.trispec_verify_attn_workspace), (self.lm_args, ts.trispec_lmhead_stats_workspace)):
            ws = ts.alloc_workspace(need(a))
            a.workspace, a.workspace_bytes = ws.data_ptr(), ws.numel()
            self.ws.append(ws)
        active = torch.zeros(B, dtype=torch.uint8, device="cuda")
        active[self.seqs] = 1
        self.active = active
        self.scan_args = ts.scan_args(self.stats, self.parent, self.tok, 0.5, ts.MODE_TARGET if target else ts.MODE_PROXY,
                                      self.out, active=active)

    def spoil(self):
        self.o.fill_(float("nan"))
        self.lse.fill_(float("nan"))
        self.mask.zero_()
        for v in list(self.stats.values()) + list(self.out.values()):
            v.zero_()

    def separate(self, stream=None):
        from paper_2601_23180_b200 import binding as ts
        ts.trispec_build_tree_mask(self.tree_args, stream)
        ts.trispec_verify_attn(self.attn_args, stream)
        ts.trispec_lmhead_stats(self.lm_args, stream)
        ts.trispec_accept_scan(self.scan_args, stream)

    def fused(self, stream=None):
        from paper_2601_23180_b200 import binding as ts
        ts.trispec_verify(self.tree_args, self.attn_args, self.lm_args, self.scan_args, stream)

    def snapshot(self):
        import torch
        torch.cuda.synchronize()
        assert int(self.status.item()) == 0
        return dict(o=self.o.view(torch.int16).clone(), lse=self.lse.view(torch.int32).clone(), mask=self.mask.clone(),
                    **{"s_" + k: v.clone() for k, v in self.stats.items()}, **{"d_" + k: v.clone() for k, v in self.out.items()})

    def attention64(self, b):
        """o of sequence b in 64 bits, [nodes][Hq][128]"""
        import torch
        L, n, Hkv = self.lens[b], self.n_nodes[b], self.kc.shape[2]
        if self.table is None:
            k, v = self.kc[b, :L], self.vc[b, :L]
        else:
            rows = self.table[b].long()
            k, v = self.kc[rows].reshape(-1, Hkv, 128)[:L], self.vc[rows].reshape(-1, Hkv, 128)[:L]
        G = self.q.shape[2] // Hkv
        k = torch.cat([k, self.kt[b, :n]]).double().repeat_interleave(G, 1)
        v = torch.cat([v, self.vt[b, :n]]).double().repeat_interleave(G, 1)
        s = torch.einsum("nhd,lhd->hnl", self.q[b, :n].double(), k) * self.scale
        bits = (self.mask[b, :n, None] >> torch.arange(n, device="cuda")) & 1
        s[:, :, L:] = s[:, :, L:].masked_fill(bits[None] == 0, float("-inf"))
        return torch.einsum("hnl,lhd->nhd", torch.softmax(s, -1), v)


def assert_same_attention(got, want):
    for k in ("o", "lse", "mask", "s_top1_idx", "d_path", "d_accept_len", "d_escalate"):
        assert bool((got[k] == want[k]).all()), k
    # sums over other ranges of the vocabulary: fp32 sums of 150000 terms, lse of about 15
    assert (got["s_lse"] - want["s_lse"]).abs().max().item() <= 1e-4


@pytest.mark.parametrize("kw", [
    dict(T=61, Hq=16, Hkv=8, cap=4096, lens=[4096]),                       # 8 splits of 8 tiles
    dict(T=61, Hq=16, Hkv=8, cap=4096, lens=[130]),                        # 3 tiles: five empty splits
    dict(T=61, Hq=16, Hkv=8, cap=4096, lens=[1000], paged=True),
    dict(T=61, Hq=16, Hkv=8, cap=4096, lens=[4033], paged=True),           # the last tile holds one key
    dict(T=61, Hq=16, Hkv=8, cap=2048, lens=[0]),                          # the tree alone
    dict(T=2, Hq=16, Hkv=16, cap=1024, lens=[777]),
    dict(T=61, Hq=64, Hkv=8, cap=2048, lens=[1999], target=True),          # four M tiles
    dict(T=9, Hq=128, Hkv=8, cap=1500, lens=[1500]),                       # 8 nodes per M tile: the second holds one
    dict(T=61, Hq=16, Hkv=8, cap=704, lens=[700, 333]),                    # 122 rows, 2 splits
    dict(T=9, Hq=32, Hkv=8, cap=1024, lens=[1000, 64, 65]),                # three sequences, 4 splits
    dict(T=61, Hq=16, Hkv=8, cap=2048, lens=[2048, 900], n_nodes=[40, 1]),  # pruned trees
    dict(T=61, Hq=64, Hkv=4, cap=2048, lens=[1024, 900], n_nodes=[40, 7]),  # M tiles without a node
    dict(T=9, Hq=16, Hkv=8, cap=1024, lens=[1000, 800, 513, 64], listed=[3, 0]),
    dict(T=61, Hq=16, Hkv=8, cap=8192, lens=[8192]),                       # 16 splits through the workspace: not in turn
    dict(T=61, Hq=16, Hkv=8, cap=16384, lens=[16000]),
])
def test_fused_pass_gives_the_attentions_own_bits(kw):
    import torch
    p = Pass(**kw)
    p.spoil()
    p.separate()
    want = p.snapshot()
    for _ in range(3):
        p.spoil()
        p.fused()
        assert_same_attention(p.snapshot(), want)
    for b in p.seqs:
        n = p.n_nodes[b]
        x, y = p.o[b, :n].double(), p.attention64(b)
        # P rounded to bf16 relative to each split's maximum, partials and the result to bf16: 2^-9 each, at most
        assert (torch.linalg.norm(x - y) / torch.linalg.norm(y)).item() <= 3 * 2.0 ** -9
