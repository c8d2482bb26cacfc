"""LM head of the pair kernels against 64-bit arithmetic at sizes where their tiles can go wrong."""
import pytest

pytestmark = pytest.mark.gpu


def _check(B, T, d, V, entropy, seed=1):
    import torch
    from paper_2601_23180_b200 import binding as ts
    scale = 3.0
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    W = torch.randn(V, d, generator=g, device="cuda", dtype=torch.bfloat16).mul_(0.8 / d ** 0.5)
    h = torch.randn(B, T, d, generator=g, device="cuda", dtype=torch.bfloat16)
    parent = torch.arange(-1, T - 1, dtype=torch.int32, device="cuda").repeat(B, 1).contiguous()
    tok = torch.randint(0, V, (B, T), generator=g, device="cuda", dtype=torch.int32)
    st = ts.alloc_stats(B, T, entropy=entropy)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    a = ts.lmhead_args(h, W, parent, tok, scale, st, dev_status=status)
    ws = ts.alloc_workspace(ts.trispec_lmhead_stats_workspace(a))
    a.workspace, a.workspace_bytes = ws.data_ptr(), ws.numel()
    ts.trispec_lmhead_stats(a)
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    W64 = W.double()
    for b in range(B):
        z = scale * (h[b].double() @ W64.T)
        lse = torch.logsumexp(z, 1)
        top = torch.topk(z, 3, dim=1)
        # fp32 accumulation of d terms and V exponentials: about 1e-6 of values of at most 40
        assert (st["lse"][b].double() - lse).abs().max().item() < 1e-4
        assert (st["max"][b].double() - top.values[:, 0]).abs().max().item() < 1e-4
        assert (st["top2_val"][b].double() - top.values[:, 1]).abs().max().item() < 1e-4
        if entropy:
            p = torch.softmax(z, 1)
            assert (st["entropy"][b].double() + (p * torch.log(p + 1e-300)).sum(1)).abs().max().item() < 1e-3
        clear = top.values[:, 0] - top.values[:, 1] > 1e-4
        assert torch.equal(st["top1_idx"][b][clear].long(), top.indices[:, 0][clear])
        clear &= top.values[:, 1] - top.values[:, 2] > 1e-4
        assert torch.equal(st["top2_idx"][b][clear].long(), top.indices[:, 1][clear])
        if T > 1:
            want = torch.exp(torch.stack([z[n - 1, tok[b, n].long()] - lse[n - 1] for n in range(1, T)]))
            assert (st["p_draft"][b][1:].double() - want).abs().max().item() < 1e-4


@pytest.mark.parametrize("B,T,V", [
    (20, 52, 30000),     # 1040 rows, 5 M tiles, 4 pairs over: slices of several W tiles
    (21, 64, 50001),     # 1344 rows, 6 M tiles of 224, 2 pairs over, an odd vocabulary
    (32, 61, 40013),     # 1952 rows, 8 M tiles
    (10, 60, 9000),      # 600 rows, 3 M tiles, a short vocabulary
])
@pytest.mark.parametrize("entropy", [False, True])
def test_tail_slices_over_several_m_tiles(B, T, V, entropy):
    _check(B, T, 64, V, entropy)


@pytest.mark.parametrize("B,T,V", [
    (3, 43, 100001),      # 129 rows: 144 columns, an odd vocabulary
    (3, 61, 100000),      # 183: 192 columns, most of a tile of each CTA's last range missing
    (32, 6, 98307),      # 192 exactly
    (1, 64, 100001),      # (64: the small-row kernel, for comparison)
    (43, 6, 98304),      # 258: two tiles of 144 columns, the second with 114 rows
    (12, 26, 100007),     # 312
    (8, 48, 100007),      # 384
    (9, 57, 98400),      # 513: three tiles of 176
    (64, 9, 98333),      # 576
])
@pytest.mark.parametrize("entropy", [False, True])
def test_rows_as_columns_of_a_pair(B, T, V, entropy):
    """From 98304 entries on, rows that would leave a quarter of an M tile empty are the N side."""
    _check(B, T, 2048, V, entropy)
