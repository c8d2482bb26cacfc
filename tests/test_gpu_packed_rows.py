"""LM head over packed rows: the rows of all active sequences lie back to back in the M tiles of the GEMM, whatever
the tree size; rows of an index list are gathered into the workspace, or read in slots of 64 per sequence
where the workspace has no room for them. Sizes around the 64 and 128 rows of the small kernel and the 256 rows of an M tile."""
import math

import numpy as np
import pytest

from oracle import trispec_oracle as orc
from paper_2601_23180_b200 import inputs as gen

pytestmark = pytest.mark.gpu


def _inputs(B, T, listed, d=192, V=3001):
    cfg = gen.small_variant(gen.CONFIGS["tiny_chain"], B=B, k=T - 1, max_depth=T - 1, d=d, V=V, rho=0.2,
                            logit_scale=3.6 / (0.02 * math.sqrt(d)), seed=B * 100 + T)
    inp = gen.make_inputs(cfg, with_attention=False)
    if listed:
        inp["seq_index"] = np.random.default_rng(B).permutation(B)[:listed].astype(np.int32)
    return cfg, inp


@pytest.mark.parametrize("B,T,listed", [
    (7, 9, 0),       # 63 rows: one N tile of the small kernel
    (8, 8, 0),       # 64
    (13, 5, 0),      # 65: the pair kernel, one M tile
    (16, 8, 0),      # 128
    (43, 3, 0),      # 129
    (17, 15, 0),     # 255
    (32, 8, 0),      # 256
    (86, 3, 0),      # 258: a second M tile with two rows
    (40, 13, 0),     # 520: 3 M tiles, two pairs left over for the tail
    (9, 9, 3),       # 27 of 81 rows: the small kernel, three slots of 16 columns
    (9, 16, 8),      # 128, gathered for the pair kernel
    (9, 17, 6),      # 102
    (20, 8, 9),      # 72: more than eight sequences, gathered
    (20, 9, 16),     # 144, gathered for the pair kernel
    (12, 61, 9),     # 549
])
@pytest.mark.parametrize("room", ["full", "slots"])
def test_lmhead_packed_rows_against_oracle(B, T, listed, room):
    import torch
    from paper_2601_23180_b200 import binding as ts
    import tests.gpu_helpers as H
    cfg, inp = _inputs(B, T, listed)
    dev = H.to_device(inp)
    seqs = list(range(B)) if not listed else [int(s) for s in inp["seq_index"]]
    st = ts.alloc_stats(B, T, entropy=True)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    a = ts.lmhead_args(dev["h"], dev["W"], dev["parent"], dev["tok"], cfg.logit_scale, st, seq_index=dev["seq_index"],
                       dev_status=status)
    need = ts.trispec_lmhead_stats_workspace(a)
    # Rows of a list are gathered where that saves M tiles, or (small kernel) where they do not fit its columns in slots
    # of a multiple of 8 for at most eight sequences.
    rows = listed * T
    gather = rows > 0 and ((rows + 255) // 256 < (listed + 3) // 4 if rows > 64
                           else listed > 8 or listed * ((T + 7) // 8 * 8) > 128)
    gathered = rows * cfg.d * 2 if gather else 0
    in_place = not gather
    if room == "slots":
        if in_place:
            pytest.skip("nothing to gather")
        need -= gathered
    ws = ts.alloc_workspace(need)
    a.workspace, a.workspace_bytes = ws.data_ptr(), need
    ts.trispec_lmhead_stats(a)
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    got = {k: v.cpu().numpy() for k, v in st.items()}
    ref = orc.lmhead_stats(inp["h"], inp["W"], inp["parent"], inp["tok"], cfg.logit_scale, seqs=seqs)
    n_tie = H.check_stats(got, ref, seqs, T)
    assert n_tie <= 0.02 * len(seqs) * T + 2
    for b in set(range(B)) - set(seqs):
        assert np.isnan(got["lse"][b]).all() and (got["top1_idx"][b] == -1).all()
    a.workspace_bytes = need - gathered - 1 if room == "full" else need - 1
    n0 = ts.launch_count()
    with pytest.raises(ts.TrispecError) as e:
        ts.trispec_lmhead_stats(a)
    assert e.value.code == 3 and ts.launch_count() == n0


@pytest.mark.parametrize("B,T,listed", [
    (13, 5, 0),      # 65 rows
    (16, 8, 0),      # 128
    (9, 25, 3),      # three slots of 32 columns
    (10, 9, 9),      # 81, gathered
])
def test_lmhead_of_up_to_128_rows_over_a_long_stream_of_weights(B, T, listed):
    """65 to 128 rows take the small kernel only where the weights are 256 MiB or more; an odd vocabulary."""
    import torch
    from paper_2601_23180_b200 import binding as ts
    d, V, scale = 896, 150001, 3.0
    g = torch.Generator(device="cuda")
    g.manual_seed(B)
    W = torch.randn(V, d, generator=g, device="cuda", dtype=torch.bfloat16).mul_(0.02)
    h = torch.randn(B, T, d, generator=g, device="cuda", dtype=torch.bfloat16)
    parent = torch.arange(-1, T - 1, dtype=torch.int32, device="cuda").repeat(B, 1).contiguous()
    tok = torch.randint(0, V, (B, T), generator=g, device="cuda", dtype=torch.int32)
    seqs = list(range(B)) if not listed else [(3 * i + 1) % B for i in range(listed)]
    index = torch.tensor(seqs, dtype=torch.int32, device="cuda") if listed else None
    st = ts.alloc_stats(B, T, entropy=True)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    a = ts.lmhead_args(h, W, parent, tok, scale, st, seq_index=index, dev_status=status)
    ws = ts.alloc_workspace(ts.trispec_lmhead_stats_workspace(a))
    a.workspace, a.workspace_bytes = ws.data_ptr(), ws.numel()
    ts.trispec_lmhead_stats(a)
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    W64 = W.double()
    for b in seqs:
        z = scale * (h[b].double() @ W64.T)
        lse = torch.logsumexp(z, 1)
        top = torch.topk(z, 3, dim=1)
        # fp32 accumulation over d = 896 and 150001 exponentials: about 1e-6 of values of about 13
        assert (st["lse"][b].double() - lse).abs().max().item() < 1e-4
        assert (st["top1_val"][b].double() - top.values[:, 0]).abs().max().item() < 1e-4
        assert (st["top2_val"][b].double() - top.values[:, 1]).abs().max().item() < 1e-4
        p = torch.softmax(z, 1)
        assert (st["entropy"][b].double() + (p * torch.log(p)).sum(1)).abs().max().item() < 1e-3
        clear = top.values[:, 0] - top.values[:, 1] > 1e-4
        assert torch.equal(st["top1_idx"][b][clear].long(), top.indices[:, 0][clear])
        clear &= top.values[:, 1] - top.values[:, 2] > 1e-4
        assert torch.equal(st["top2_idx"][b][clear].long(), top.indices[:, 1][clear])
        want = torch.stack([z[n - 1, tok[b, n].long()] for n in range(1, T)])
        assert (st["draft_logit"][b, 1:].double() - want).abs().max().item() < 1e-4


@pytest.mark.parametrize("B,k,tree,L,V,d,form", [
    (1, 60, "random", 1000, 40000, 2048, None),           # two KV splits beside the LM head
    (3, 8, "chain", 500, 40000, 2048, "side_by_side"),    # three sequences, 27 rows: unsplit
    (2, 60, "random", 700, 70000, 2048, "side_by_side"),  # 122 rows
    (1, 60, "random", 4096, 120000, 2048, "lm_first"),    # 8 CTAs of 65 tiles beside it instead of 64 after it
])
def test_few_row_pass_with_its_attention_beside_the_lm_head(B, k, tree, L, V, d, form):
    import torch
    from paper_2601_23180_b200 import binding as ts, runner
    cfg = gen.small_variant(gen.CONFIGS["proxy_tree"], B=B, k=k, tree=tree, max_depth=min(k, 6), L=L, V=V, d=d, seed=5,
                            logit_scale=3.6 / (0.02 * math.sqrt(d)))
    pas = runner.VerifyPass(cfg, gen.make_inputs(cfg))
    if form:
        assert ts.trispec_verify_plan(pas.attn_args, pas.lm_args, pas.scan_args) == form
    ts.trispec_build_tree_mask(pas.tree_args)
    ts.trispec_verify_attn(pas.attn_args)
    ts.trispec_lmhead_stats(pas.lm_args)
    ts.trispec_accept_scan(pas.scan_args)
    torch.cuda.synchronize()
    want = pas.o.float().clone(), pas.stats["lse"].clone(), pas.stats["top1_idx"].clone(), pas.scan_out["path"].clone()
    for _ in range(5):
        pas.o.fill_(float("nan")); pas.mask.zero_(); pas.stats["lse"].zero_(); pas.stats["top1_idx"].fill_(-7)
        pas.scan_out["path"].fill_(-9)
        pas.run()
        got = pas.o.float().clone(), pas.stats["lse"].clone(), pas.stats["top1_idx"].clone(), pas.scan_out["path"].clone()
        torch.cuda.synchronize()
        # two bf16 roundings of outputs of at most about 4 (half a step is 8e-3), as in the parity tests
        assert (got[0] - want[0]).abs().max().item() <= 2e-2
        assert (got[1] - want[1]).abs().max().item() <= 1e-4      # fp32 sums in another order, lse of about 30
        assert torch.equal(got[2], want[2]) and torch.equal(got[3], want[3])
