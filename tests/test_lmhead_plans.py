"""What the LM head asks for and which kernel a call takes, seen from the host: without a device the planner assumes
148 SMs."""
import pytest

from paper_2601_23180_b200 import binding as ts
from paper_2601_23180_b200 import inputs as gen


def _lm(B, T, d, V, listed=0):
    a = ts.LmheadArgs()
    a.B, a.T, a.d, a.V, a.logit_scale = B, T, d, V, 1.0
    a.B_active, a.seq_index = listed, 1 if listed else None
    return a


@pytest.mark.parametrize("B,T,d,V", [
    (9, 9, 2048, 32000),       # 81 packed rows: one M tile
    (12, 21, 2048, 32000),     # 252: one M tile of 256 rows, whose partials would take 74 ranges
    (12, 10, 2048, 151936),    # 120 rows over a long W: the small-row kernel
])
def test_several_sequences_ask_for_the_workspace_of_their_slots_and_no_more(B, T, d, V):
    # 9 to 12 sequences in slots of 64 rows are three M tiles: 24 ranges x 3 x 256 rows x 32 bytes
    assert ts.trispec_lmhead_stats_workspace(_lm(B, T, d, V)) == 24 * 3 * 256 * 32
    # with an index list, room for the gathered rows comes on top of it
    rows = B * T * d * 2
    assert ts.trispec_lmhead_stats_workspace(_lm(B, T, d, V, B)) == 24 * 3 * 256 * 32 + rows


def test_pass_form_asks_which_kernel_the_lm_head_takes():
    """Ten listed sequences of six nodes are gathered for the small-row kernel; a workspace that was sized without a
    list leaves them in slots in the pair kernel, which takes every SM: nothing runs beside it."""
    cfg = gen.small_variant(gen.CONFIGS["tiny_chain"], B=12, L=256, Hq=8, Hkv=1)
    t = ts.AttnArgs()
    t.B, t.T, t.Hq, t.Hkv, t.D, t.scale = cfg.B, 6, cfg.Hq, cfg.Hkv, cfg.D, 1.0
    t.kv_layout, t.Lmax, t.B_active, t.seq_index = ts.KV_CONTIGUOUS, cfg.L, 10, 1
    lm = _lm(12, 6, 2048, 60000, 10)
    lm.workspace_bytes = ts.trispec_lmhead_stats_workspace(lm)
    assert ts.trispec_verify_plan(t, lm) == "side_by_side"
    lm.workspace_bytes = ts.trispec_lmhead_stats_workspace(_lm(12, 6, 2048, 60000))
    assert ts.trispec_verify_plan(t, lm) == "attention_first"
