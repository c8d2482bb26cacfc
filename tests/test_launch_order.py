"""How a call's launches are ordered behind earlier work, seen from the requests to the CUDA runtime."""
from tests.host_launches import requests

EVERY_CALL = """
S = 77                                            # the caller's stream
forms = dict(one_launch=dict(), in_turn=dict(T=61, cap=4096, V=151936), two_streams=dict(T=9, Hq=8, Hkv=1, cap=8192),
             lm_first=dict(T=61, cap=8192, V=151936), batch=dict(B=8, T=61, cap=4096), pieces=dict(B=40, T=61, cap=32768),
             listed=dict(B=12, T=61, listed=5, cap=700, V=151936), columns=dict(B=3, T=61, cap=700, d=5120, V=151936), many=dict(B=3000, T=9, cap=64))
for name, kw in forms.items():
    p = Args(**kw)
    structs = (r(p.tree), r(p.attn), r(p.lm), r(p.scan), S)
    call("verify_" + name, lib.trispec_verify(*structs))
    call("host_" + name, lib.trispec_verify_host(r(ts.HostIO()), *structs))
    call("mask_" + name, lib.trispec_build_tree_mask(r(p.tree), S))
    call("attn_" + name, lib.trispec_verify_attn(r(p.attn), S))
    call("lmhead_" + name, lib.trispec_lmhead_stats(r(p.lm), S))
    call("scan_" + name, lib.trispec_accept_scan(r(p.scan), S))
    if name == "one_launch":
        call("noalloc", lib.trispec_lmhead_stats_noalloc(r(p.lm), S))
    c = ts.CommitArgs()
    c.B, c.T, c.Hkv, c.D, c.kv_layout, c.Lmax = p.attn.B, p.attn.T, p.attn.Hkv, 128, ts.KV_CONTIGUOUS, p.attn.Lmax
    for f in ("k_tree", "v_tree", "k_cache", "v_cache", "ctx_len"):
        setattr(c, f, getattr(p.attn, f))
    c.path, c.accept_len, c.ctx_len_out = p.scan.path, p.scan.accept_len, p.new()
    call("commit_" + name, lib.trispec_commit_kv(r(c), S))
    u = ts.PruneArgs()
    u.B, u.T, u.parent, u.tok, u.mask = p.tree.B, p.tree.T, p.tree.parent, p.lm.tok, p.tree.mask
    for f in ("root", "n_keep", "node_map", "parent_out", "tok_out", "mask_out"):
        setattr(u, f, p.new())
    call("prune_" + name, lib.trispec_prune_tree(r(u), S))
    b = ts.SampleArgs()
    b.B, b.T, b.d, b.V, b.logit_scale = p.lm.B, p.lm.T, p.lm.d, p.lm.V, 1.0
    b.h, b.W, b.last_node, b.bonus_tok = p.lm.h, p.lm.W, p.scan.last_node, p.scan.bonus_tok
    b.workspace, b.workspace_bytes = p.new(), ts.trispec_sample_bonus_workspace(b)
    call("sample_" + name, lib.trispec_sample_bonus(r(b), S))
"""


def test_the_first_kernel_of_every_call_is_an_ordinary_launch(tmp_path):
    """A programmatic dependent waits for the kernel right ahead of it; a call's first kernel has to wait for everything
    on its stream, whatever the caller put there last."""
    calls = requests(tmp_path, EVERY_CALL)
    assert len(calls) == 9 * 9 + 1
    kernels = set()
    for name, log in calls.items():
        launches = [x for what, _, x in log if what == "launch"]
        kernels |= {x.kernel for x in launches}
        assert launches, name
        for stream in {x.stream for x in launches}:
            own = [x for x in launches if x.stream == stream]
            assert not own[0].dependent, (name, own[0].kernel)
        # the kernels inside a call are dependents of each other
        if name.startswith("verify_") and "streams" not in name:
            assert all(x.dependent for x in launches[1:]), name
    for part in ("rows_beside", "lmhead_cols", "lmhead_gemm", "attn_pieces_kernel", "attn_split", "attn_merge", "tree_mask_block",
                 "esc_compact", "sample_gather", "pack_rows", "prune_tree", "kv_commit_kernel"):
        assert any(part in k for k in kernels), part


BESIDE = """
for name, kw in dict(one_each_would_do=dict(d=8192), two_each=dict(d=4096), one_each=dict(B=3, d=8192),
                     second_stream=dict(Hq=8, Hkv=1, cap=8192)).items():
    p = Args(**dict(kw, V=15872))
    call(name + ":%d" % ts.trispec_verify_beside(p.attn, p.lm, p.scan), lib.trispec_verify(r(p.tree), r(p.attn), r(p.lm), r(p.scan), 77))
"""


def test_the_answer_beside_the_lm_head_is_the_number_of_ctas_launched(tmp_path):
    """992 units of 16 vocabulary entries are 124 ranges of 8 wherever the LM head is left 124 to 141 SMs."""
    for name, log in requests(tmp_path, BESIDE).items():
        launches = [x for what, _, x in log if what == "launch"]
        rows = next(x for x in launches if "lmhead_rows" in x.kernel)
        attn = [x.grid for x in launches if "attn_split" in x.kernel]
        assert ("rows_beside" in rows.kernel) != bool(attn)
        assert int(name.split(":")[1]) == (attn[0] if attn else rows.grid - 124) > 0, name


SHARED = """
for name in ("apart", "depth_in_lse", "parents_in_o", "depth_in_n_nodes", "other_mask", "other_batch"):
    p = Args(B=2, V=151936)
    if name == "depth_in_lse": p.tree.depth = p.attn.lse
    if name == "parents_in_o": p.tree.parent = p.attn.o + 64
    if name == "depth_in_n_nodes": p.attn.n_nodes = p.tree.depth
    if name == "other_mask": p.attn.mask = p.new()
    if name == "other_batch": p.tree.B = 3
    call(name, lib.trispec_verify(r(p.tree), r(p.attn), r(p.lm), r(p.scan), 77))
"""


def test_masks_come_first_where_the_tree_step_shares_memory_with_the_attention(tmp_path):
    """In the launch that has masks and attention they run at the same time: only where neither writes what the other touches."""
    for name, log in requests(tmp_path, SHARED).items():
        kernels = [x.kernel for what, _, x in log if what == "launch"]
        assert ["tree_mask" in k for k in kernels].index(False) == (0 if name == "apart" else 1), name
        assert any("rows_beside" in k for k in kernels), name


COLUMNS = """
for rows, d, V, cols in ((150, 2048, 98304, 1), (150, 2048, 98303, 0), (150, 1984, 151936, 0), (312, 4096, 128256, 1), (386, 4096, 128256, 0),
                         (513, 5120, 98304, 1), (576, 2048, 65600, 0), (784, 4096, 151936, 0)):
    p = Args(B=rows, T=1, d=d, V=V)
    call("%d_%d_%d:%d" % (rows, d, V, cols), lib.trispec_lmhead_stats(r(p.lm), 77))
"""


def test_which_lm_heads_take_rows_as_columns(tmp_path):
    for name, log in requests(tmp_path, COLUMNS).items():
        kernels = [x.kernel for what, _, x in log if what == "launch"]
        assert any("lmhead_cols" in k for k in kernels) == (name[-1] == "1"), name
