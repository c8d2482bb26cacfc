"""What the fused passes decide on the host before anything is launched; addresses are never followed."""
import ctypes

import pytest

from paper_2601_23180_b200 import binding as ts


class Args:
    """Argument structs of one pass whose buffers lie 256 MiB apart at made-up addresses."""

    def __init__(self, B=1, T=9, Hq=16, Hkv=8, cap=512, d=2048, V=32000, listed=0):
        self.at = 1 << 40
        t, a, l, s = ts.TreeArgs(), ts.AttnArgs(), ts.LmheadArgs(), ts.ScanArgs()
        t.B, t.T, t.parent, t.mask, t.depth = B, T, self.new(), self.new(), self.new()
        a.B, a.T, a.Hq, a.Hkv, a.D, a.scale = B, T, Hq, Hkv, 128, 0.1
        a.kv_layout, a.Lmax = ts.KV_CONTIGUOUS, cap
        for f in ("q", "k_tree", "v_tree", "k_cache", "v_cache", "ctx_len", "o", "lse"):
            setattr(a, f, self.new())
        a.mask = t.mask
        l.B, l.T, l.d, l.V, l.logit_scale = B, T, d, V, 1.0
        l.h, l.W, l.parent, l.tok = self.new(), self.new(), t.parent, self.new()
        for f in ("max", "lse", "top1_val", "top2_val", "p_top1", "p_top2", "top1_idx", "top2_idx", "draft_logit", "p_draft"):
            setattr(l.out, f, self.new())
        s.B, s.T, s.lam, s.parent, s.tok, s.stats = B, T, 0.5, t.parent, l.tok, l.out
        for f in ("accept_len", "bonus_tok", "path", "last_node", "escalate", "n_escalated", "esc_index"):
            setattr(s, f, self.new())
        if listed:
            a.seq_index = l.seq_index = self.new()
            a.B_active = l.B_active = listed
        a.workspace, a.workspace_bytes = self.new(), ts.trispec_verify_attn_workspace(a)
        l.workspace, l.workspace_bytes = self.new(), ts.trispec_lmhead_stats_workspace(l)
        self.tree, self.attn, self.lm, self.scan = t, a, l, s

    def new(self):
        self.at += 256 << 20
        return self.at

    def call(self, host):
        lib, r = ts._lib, ctypes.byref
        structs = (r(self.tree), r(self.attn), r(self.lm), r(self.scan), None)
        return lib.trispec_verify_host(r(ts.HostIO()), *structs) if host else lib.trispec_verify(*structs)

    def form(self):
        return ts.trispec_verify_plan(self.attn, self.lm, self.scan)


@pytest.mark.parametrize("host", [False, True])
@pytest.mark.parametrize("shape", [dict(), dict(B=8, T=61, cap=4096), dict(V=151936, T=61, cap=4096)],
                         ids=["beside", "attention_first", "in_turn"])
@pytest.mark.parametrize("step,field,value,code", [
    ("tree", "mask", None, 1), ("attn", "o", None, 1), ("attn", "scale", 0.0, 1), ("attn", "q", 4096 + 8, 1),
    ("attn", "D", 64, 2), ("lm", "W", None, 1), ("lm", "workspace_bytes", 256, 3), ("lm", "d", 100, 2),
    ("scan", "path", None, 1), ("scan", "criterion", 9, 1), ("scan", "u_accept", 4096, 1),
])
def test_an_argument_error_of_any_step_is_found_before_the_first_launch(host, shape, step, field, value, code):
    p = Args(**shape)
    setattr(getattr(p, step), field, value)
    n0 = ts.launch_count()
    assert p.call(host) == code
    assert ts.launch_count() == n0


@pytest.mark.parametrize("B", [1, 4])
def test_a_fused_pass_asks_for_the_attentions_workspace(B):
    """The split plan of a long context merges through the workspace, whatever form the pass would take."""
    p = Args(B=B, T=9, Hq=8, Hkv=1, cap=16384, V=151936)
    assert p.attn.workspace_bytes > 0
    p.attn.workspace_bytes -= 1
    assert p.call(False) == 3 and p.call(True) == 3
    p.attn.workspace_bytes += 1
    p.attn.workspace = None
    assert p.call(False) == 1


@pytest.mark.parametrize("shape", [dict(), dict(B=4, listed=1), dict(B=3, V=151936)])
def test_steps_that_share_written_memory_run_in_stream_order(shape):
    in_order = "attention_first" if shape.get("B") == 3 else "lm_first"
    p = Args(**shape)
    assert p.form() == "side_by_side"
    n = p.scan.B * 4
    if p.attn.seq_index:
        for at in (p.attn.seq_index, p.attn.seq_index - n + 4, p.attn.seq_index - 4):
            p.scan.esc_index = at
            assert p.form() == (in_order if at + n > p.attn.seq_index else "side_by_side"), at
        p.scan.esc_index = p.attn.seq_index + 4                 # behind the one listed entry
        assert p.form() == "side_by_side"
    p.lm.workspace, keep = p.attn.o, p.lm.workspace
    assert p.form() == in_order
    p.lm.workspace = keep
    p.scan.path, keep = p.attn.ctx_len, p.scan.path
    assert p.form() == in_order
    p.scan.path = keep
    p.scan.last_node, keep = p.attn.mask + 8, p.scan.last_node
    assert p.form() == in_order
    p.scan.last_node = keep
    assert p.form() == "side_by_side"


def test_a_workspace_shared_by_the_attention_and_the_lm_head():
    p = Args(B=1, T=9, Hq=8, Hkv=1, cap=8192)                   # 16 splits through the workspace, 16 CTAs
    assert p.attn.workspace_bytes > 0 and p.form() == "side_by_side"
    p.lm.workspace = p.attn.workspace
    assert p.form() == "lm_first"
    p.lm.workspace = p.attn.workspace + p.attn.workspace_bytes  # one buffer, one part each
    assert p.form() == "side_by_side"


@pytest.mark.parametrize("shape,form,ctas", [
    (dict(), "side_by_side", 16),                                            # the attention's own 8 x 2 splits
    (dict(V=151936), "side_by_side", 16),                                    # a long W: a pair of CTAs per KV head
    (dict(T=61, cap=4096, V=151936), "lm_first", 16),                        # 8 x 8 splits in turn, in pairs
    (dict(T=61, cap=8192, V=151936), "lm_first", 0),                         # 16 splits through the workspace
    (dict(T=61, Hq=64, cap=8192, d=5120, V=151936), "lm_first", 32),
    (dict(B=3, V=151936), "side_by_side", 24),
    (dict(B=2, T=61, cap=704, V=151936), "side_by_side", 16),
    (dict(B=8, T=61, cap=4096, V=151936), "attention_first", 0),
    (dict(B=12, T=5, listed=9, cap=256, V=151936), "attention_first", 0),    # 72 CTAs
])
def test_the_plan_tells_what_runs_beside_the_lm_head(shape, form, ctas):
    p = Args(**shape)
    assert p.form() == form
    assert ts.trispec_verify_beside(p.attn, p.lm, p.scan) == ctas
    p.scan.path = p.attn.ctx_len
    assert ts.trispec_verify_beside(p.attn, p.lm, p.scan) == 0
    assert ts.trispec_verify_beside(None, p.lm, p.scan) == 0
