"""LM head with the least workspace that a call may bring, whatever way its rows are read."""
import math

import numpy as np
import pytest

from oracle import trispec_oracle as orc
from paper_2601_23180_b200 import inputs as gen

pytestmark = pytest.mark.gpu


def _call(B, T, listed, d, V, seed=7):
    import torch
    import tests.gpu_helpers as H
    from paper_2601_23180_b200 import binding as ts
    cfg = gen.small_variant(gen.CONFIGS["tiny_chain"], B=B, k=T - 1, max_depth=T - 1, d=d, V=V, rho=0.2,
                            logit_scale=3.6 / (0.02 * math.sqrt(d)), seed=seed)
    inp = gen.make_inputs(cfg, with_attention=False)
    if listed:
        inp["seq_index"] = np.random.default_rng(B).permutation(B)[:listed].astype(np.int32)
    dev = H.to_device(inp)
    st = ts.alloc_stats(B, T, entropy=True)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    a = ts.lmhead_args(dev["h"], dev["W"], dev["parent"], dev["tok"], cfg.logit_scale, st, seq_index=dev["seq_index"],
                       dev_status=status)
    a._held += (dev,)
    return cfg, inp, a, st, status


def _check(cfg, inp, st, status, T, B):
    import tests.gpu_helpers as H
    assert int(status.item()) == 0
    seqs = list(range(B)) if inp.get("seq_index") is None else [int(s) for s in inp["seq_index"]]
    got = {k: v.cpu().numpy() for k, v in st.items()}
    ref = orc.lmhead_stats(inp["h"], inp["W"], inp["parent"], inp["tok"], cfg.logit_scale, seqs=seqs)
    assert H.check_stats(got, ref, seqs, T) <= 0.02 * len(seqs) * T + 2
    for b in set(range(B)) - set(seqs):
        assert np.isnan(got["lse"][b]).all() and (got["top1_idx"][b] == -1).all()


@pytest.mark.parametrize("B,T,d,V", [
    (12, 21, 192, 3001),       # 252 packed rows: 72 vocabulary ranges instead of 74
    (9, 9, 192, 3001),
    (33, 31, 64, 20011),       # 1023: four M tiles of 256, nine in slots
    (24, 53, 64, 20011),       # 1272: five M tiles, whose tail pairs have to fit as well
    (12, 10, 2048, 65552),     # 120 rows over 256 MiB of W: the small-row kernel with 144 ranges
])
def test_lmhead_with_the_workspace_of_the_slots(B, T, d, V):
    import torch
    from paper_2601_23180_b200 import binding as ts
    cfg, inp, a, st, status = _call(B, T, 0, d, V)
    need = ts.trispec_lmhead_stats_workspace(a)
    ws = torch.full((need + 4096,), 0x5A, dtype=torch.uint8, device="cuda")
    a.workspace, a.workspace_bytes = ws.data_ptr(), need
    ts.trispec_lmhead_stats(a)
    torch.cuda.synchronize()
    assert (ws[need:] == 0x5A).all()
    _check(cfg, inp, st, status, T, B)


@pytest.mark.parametrize("B,T,listed", [(20, 5, 12), (12, 6, 10)])     # 60 rows of more than eight sequences
@pytest.mark.parametrize("room", ["gathered", "slots"])
def test_few_listed_rows_with_and_without_room_to_gather(B, T, listed, room):
    import torch
    from paper_2601_23180_b200 import binding as ts
    cfg, inp, a, st, status = _call(B, T, listed, 192, 3001)
    need = ts.trispec_lmhead_stats_workspace(a) - (0 if room == "gathered" else listed * T * 192 * 2)
    ws = torch.full((need + 4096,), 0x5A, dtype=torch.uint8, device="cuda")
    a.workspace, a.workspace_bytes = ws.data_ptr(), need
    n0 = ts.launch_count()
    ts.trispec_lmhead_stats(a)
    torch.cuda.synchronize()
    assert ts.launch_count() - n0 == (3 if room == "gathered" else 2)
    assert (ws[need:] == 0x5A).all()
    _check(cfg, inp, st, status, T, B)


@pytest.mark.parametrize("room", ["gathered", "slots"])
def test_fused_pass_of_listed_rows_with_and_without_room_to_gather(room):
    import torch
    from paper_2601_23180_b200 import binding as ts
    from tests.test_gpu_beside import Pass, assert_same_attention
    p = Pass(T=6, Hq=8, Hkv=1, cap=256, lens=[200 + i for i in range(12)], listed=[11, 3, 0, 7, 5, 1, 9, 2, 8, 4], V=60000)
    if room == "slots":
        p.lm_args.workspace_bytes -= 60 * 2048 * 2
    assert ts.trispec_verify_plan(p.attn_args, p.lm_args, p.scan_args) == ("side_by_side" if room == "gathered" else
                                                                         "attention_first")
    p.spoil()
    p.separate()
    want = p.snapshot()
    for _ in range(3):
        p.spoil()
        p.fused()
        assert_same_attention(p.snapshot(), want)


@pytest.mark.parametrize("B,T,listed,launches", [
    (8, 9, 7, 3),      # 63 rows, but 112 columns in slots: gathered, over a short W
    (9, 12, 5, 3),     # 60 rows, 80 columns
    (9, 16, 4, 2),     # 64 rows, 64 columns: read in slots
])
def test_slots_of_the_small_row_kernel_are_counted_in_columns(B, T, listed, launches):
    import torch
    from paper_2601_23180_b200 import binding as ts
    cfg, inp, a, st, status = _call(B, T, listed, 192, 3001)
    ws = ts.alloc_workspace(ts.trispec_lmhead_stats_workspace(a))
    a.workspace, a.workspace_bytes = ws.data_ptr(), ws.numel()
    n0 = ts.launch_count()
    ts.trispec_lmhead_stats(a)
    torch.cuda.synchronize()
    assert ts.launch_count() - n0 == launches
    _check(cfg, inp, st, status, T, B)
