"""The fused pass of few rows, whose attention runs beside the LM head: in its launch, in one or two CTAs per (sequence, KV
head, M tile) that take the splits of the attention's own plan in turn, or by that plan on the second stream of the caller's
stream; the same bits as the attention called by itself, captured or not. The host-buffer pass always takes the second stream."""
import math

import pytest

pytestmark = pytest.mark.gpu


class Pass:
    """One pass with inputs drawn on the GPU. Capacity `cap` tokens per sequence, lengths `lens`."""

    def __init__(self, T, Hq, Hkv, cap, lens, listed=None, n_nodes=None, paged=False, d=2048, V=151936, seed=3, target=False,
                 entropy=True):
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
        self.seqs = list(range(B)) if listed is None else [x for x in listed if 0 <= x < B]
        self.index = None if listed is None else i32(listed)
        self.nodes = None if n_nodes is None else i32(n_nodes)
        self.n_nodes = n_nodes or [T] * B
        self.status = torch.zeros(1, dtype=torch.int32, device="cuda")
        self.mask = torch.zeros((B, T), dtype=torch.int64, device="cuda")
        self.depth = torch.zeros((B, T), dtype=torch.int32, device="cuda")
        self.o = torch.zeros((B, T, Hq, 128), dtype=torch.bfloat16, device="cuda")
        self.lse = torch.zeros((B, Hq, T), dtype=torch.float32, device="cuda")
        self.stats, self.out = ts.alloc_stats(B, T, entropy=entropy), ts.alloc_scan_out(B, T)
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
        self.depth.fill_(-7)
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

    def from_host(self, stream=None):
        """The pass with its per-round inputs in pinned memory; the device copies are spoiled first."""
        import torch
        from paper_2601_23180_b200 import binding as ts
        names = dict(parent=self.parent, tok=self.tok, h=self.h, q=self.q, k_tree=self.kt, v_tree=self.vt)
        if not hasattr(self, "pinned"):
            self.pinned = {n: t.cpu().pin_memory() for n, t in names.items()}
            self.back = {n: torch.zeros(self.out[n].shape, dtype=self.out[n].dtype).pin_memory()
                         for n in ("accept_len", "bonus_tok", "last_node", "path", "escalate")}
            self.io = ts.host_io(**self.pinned, **self.back)
        with torch.cuda.stream(stream):
            for t in names.values():
                t.zero_()
        ts.trispec_verify_host(self.io, self.tree_args, self.attn_args, self.lm_args, self.scan_args, stream)

    def snapshot(self, status=0):
        import torch
        torch.cuda.synchronize()
        assert int(self.status.item()) == status
        return dict(o=self.o.view(torch.int16).clone(), lse=self.lse.view(torch.int32).clone(), mask=self.mask.clone(),
                    depth=self.depth.clone(),
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
    for k in ("o", "lse", "mask", "depth", "s_top1_idx", "d_path", "d_accept_len", "d_escalate"):
        assert bool((got[k] == want[k]).all()), k
    # sums over other ranges of the vocabulary: fp32 sums of 150000 terms, lse of about 15
    assert (got["s_lse"] - want["s_lse"]).abs().max().item() <= 1e-4
    if "s_entropy" in want:                        # and E[z] of values of up to 40 on top of it
        assert (got["s_entropy"] - want["s_entropy"]).abs().max().item() <= 1e-3


def launches(call, *args):
    from paper_2601_23180_b200 import binding as ts
    n0 = ts.launch_count()
    call(*args)
    return ts.launch_count() - n0


# launches that a fused pass saves: masks, attention and LM head in one; the attention and the LM head; none
ONE_LAUNCH, MASKS_APART, SECOND_STREAM = 2, 1, 0


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
    dict(T=9, Hq=16, Hkv=8, cap=512, lens=[512], d=4096, V=16000),         # 16 + 125 CTAs in clusters of two
    dict(T=9, Hq=16, Hkv=8, cap=512, lens=[500], d=4096, V=16000, entropy=False),
    dict(T=61, Hq=16, Hkv=8, cap=8192, lens=[8192]),                       # 16 splits through the workspace: not in turn
    dict(T=61, Hq=16, Hkv=8, cap=16384, lens=[16000]),
])
def test_fused_pass_gives_the_attentions_own_bits(kw):
    import torch
    from paper_2601_23180_b200 import binding as ts
    p = Pass(**kw)
    per_tile = min(64, 128 * kw["Hkv"] // kw["Hq"])
    ctas = len(p.seqs) * kw["Hkv"] * ((kw["T"] + per_tile - 1) // per_tile)
    in_turn = ctas * (2 if 4 * ctas <= 148 // 4 else 1)                    # (every plan here has two splits or more)
    assert ts.trispec_verify_beside(p.attn_args, p.lm_args, p.scan_args) == (in_turn if kw["cap"] <= 4096 and ctas <= 148 // 4 else 0)
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


CHAINS = dict(T=9, Hq=32, Hkv=8, cap=256, lens=[256, 100, 31], d=2048, V=40000)      # 27 rows, 24 CTAs
ONE = dict(T=9, Hq=16, Hkv=8, cap=512, lens=[512], d=2048, V=32000)
TWO = dict(T=9, Hq=8, Hkv=1, cap=8192, lens=[8000], d=2048, V=32000)                 # 16 splits through the workspace


def _want(p):
    p.spoil()
    p.separate()
    return p.snapshot()


@pytest.mark.parametrize("call,kw,saved", [("fused", CHAINS, ONE_LAUNCH), ("from_host", CHAINS, SECOND_STREAM),
                                           ("fused", TWO, SECOND_STREAM), ("from_host", TWO, SECOND_STREAM)])
def test_a_pass_does_not_wait_for_another_callers_stream(call, kw, saved):
    import torch
    a, b = Pass(**kw), Pass(**dict(kw, seed=4))
    assert launches(a.separate) - launches(getattr(a, call)) == saved
    sa, sb = torch.cuda.Stream(), torch.cuda.Stream()
    want = [_want(a), _want(b)]
    for p, s in ((a, sa), (b, sb)):
        getattr(p, call)(s)
        torch.cuda.synchronize()
        p.spoil()
    torch.cuda.synchronize()
    reached = torch.cuda.Event()
    with torch.cuda.stream(sa):
        torch.cuda._sleep(400_000_000)             # about 0.2 s
        reached.record()
    getattr(a, call)(sa)
    getattr(b, call)(sb)
    sb.synchronize()
    assert not reached.query()                     # b's pass is done and a's has not begun
    got = [a.snapshot(), b.snapshot()]
    assert_same_attention(got[0], want[0])
    assert_same_attention(got[1], want[1])


@pytest.mark.parametrize("call,kw,saved", [
    ("fused", CHAINS, ONE_LAUNCH), ("fused", ONE, ONE_LAUNCH), ("fused", dict(T=61, Hq=16, Hkv=8, cap=4096, lens=[4096]), ONE_LAUNCH),
    ("fused", TWO, SECOND_STREAM), ("from_host", CHAINS, SECOND_STREAM), ("from_host", TWO, SECOND_STREAM),
])
def test_captured_pass_beside_an_eager_one(call, kw, saved):
    """A pass under capture, and between two of its calls an eager pass on another stream: neither disturbs the other."""
    import torch
    p, q = Pass(**kw), Pass(**dict(TWO if kw is TWO else CHAINS, seed=4))
    want_p, want_q = _want(p), _want(q)
    sp, sq = torch.cuda.Stream(), torch.cuda.Stream()
    for x, s in ((p, sp), (q, sq)):
        assert launches(x.separate, s) - launches(getattr(x, call), s) == saved
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    q.spoil()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph, stream=sp):
        getattr(p, call)(sp)
        getattr(q, call)(sq)
        getattr(p, call)(sp)
    assert_same_attention(q.snapshot(), want_q)
    for _ in range(3):
        p.spoil()
        torch.cuda.synchronize()
        graph.replay()
        assert_same_attention(p.snapshot(), want_p)
    p.spoil()
    torch.cuda.synchronize()
    getattr(p, call)(sp)                                    # the stream's second stream is usable again after the capture
    assert_same_attention(p.snapshot(), want_p)
    first = torch.cuda.CUDAGraph()
    fresh = torch.cuda.Stream()                    # a stream that the library meets under capture
    with torch.cuda.graph(first, stream=fresh):
        getattr(p, call)(fresh)
    p.spoil()
    torch.cuda.synchronize()
    first.replay()
    graph.replay()
    assert_same_attention(p.snapshot(), want_p)
    del graph, first


def test_more_busy_streams_than_second_streams():
    import torch
    tiny = dict(T=9, Hq=8, Hkv=8, cap=128, lens=[100], d=64, V=3000)
    passes = [Pass(**dict(tiny, seed=i)) for i in range(20)]
    want = [_want(p) for p in passes]
    assert launches(passes[0].separate) - launches(passes[0].fused) == SECOND_STREAM
    for rounds in range(2):
        for p in passes:
            p.spoil()
        torch.cuda.synchronize()
        gate, opened = torch.cuda.Stream(), torch.cuda.Event()
        with torch.cuda.stream(gate):
            torch.cuda._sleep(20_000_000)
            opened.record()
        streams = [torch.cuda.Stream() for _ in passes]
        for p, s in zip(passes, streams):
            s.wait_event(opened)                   # all twenty are pending at once
            p.fused(s)
        torch.cuda.synchronize()
        for p, w in zip(passes, want):
            assert_same_attention(p.snapshot(), w)


def test_threads_on_streams_of_their_own_and_on_a_shared_one():
    import threading
    import torch
    passes = [Pass(**dict(kw, seed=i)) for i, kw in enumerate((CHAINS, ONE, CHAINS, ONE, TWO, TWO))]
    want = [_want(p) for p in passes]
    shared = torch.cuda.Stream()
    streams = [torch.cuda.Stream(), torch.cuda.Stream(), shared, shared, torch.cuda.Stream(), shared]
    for p in passes:
        p.spoil()
    torch.cuda.synchronize()
    errors = []

    def work(p, s, call):
        try:
            for _ in range(40):
                getattr(p, call)(s)
        except Exception as e:                     # (reported by the main thread)
            errors.append(e)

    threads = [threading.Thread(target=work, args=(p, s, c))
               for p, s, c in zip(passes, streams, ("fused", "from_host", "from_host", "fused", "fused", "fused"))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors
    for p, w in zip(passes, want):
        assert_same_attention(p.snapshot(), w)


@pytest.mark.parametrize("kw", [CHAINS, dict(CHAINS, listed=[2, 0]), ONE, dict(T=61, Hq=16, Hkv=8, cap=704, lens=[700, 333])])
def test_host_buffer_pass_of_several_sequences(kw):
    import torch
    p = Pass(**kw)
    want = _want(p)
    for s in (torch.cuda.current_stream(), torch.cuda.Stream()):
        for _ in range(3):
            p.spoil()
            torch.cuda.synchronize()
            p.from_host(s)
            assert_same_attention(p.snapshot(), want)
            for n, t in p.back.items():
                assert torch.equal(t, p.out[n].cpu()), n


@pytest.mark.parametrize("what", ["workspace", "list"])
def test_pass_whose_steps_share_memory_runs_in_order(what):
    """One workspace for both steps; the escalation list written one entry before the list that the attention reads."""
    import torch
    from paper_2601_23180_b200 import binding as ts
    if what == "workspace":
        p = Pass(T=9, Hq=8, Hkv=1, cap=8192, lens=[8000], V=32000)
        ws = ts.alloc_workspace(max(p.attn_args.workspace_bytes, p.lm_args.workspace_bytes))
        for a in (p.attn_args, p.lm_args):
            a.workspace, a.workspace_bytes = ws.data_ptr(), ws.numel()
    else:
        p = Pass(**dict(CHAINS, listed=[2, 0]))
        buf = torch.tensor([-1, 2, 0, -1], dtype=torch.int32, device="cuda")
        for a in (p.attn_args, p.lm_args):
            a.seq_index = buf[1:].data_ptr()
        p.scan_args.esc_index = buf.data_ptr()
    want = None
    for call in (p.separate, p.fused, p.fused, p.fused):
        p.spoil()
        if what == "list":
            buf.copy_(torch.tensor([-1, 2, 0, -1], dtype=torch.int32))
        call()
        got = p.snapshot()
        if want is not None:
            assert_same_attention(got, want)
        want = want or got
    if what == "list":
        assert int(p.out["n_escalated"].item()) == int((buf[:3] >= 0).sum().item())


@pytest.mark.parametrize("kw,plan,room", [
    (dict(T=9, Hq=32, Hkv=8, cap=256, lens=[256, 100, 31, 200], listed=[2, -1, 0, 4], V=40000), None, "full"),
    (dict(T=6, Hq=8, Hkv=1, cap=256, lens=[200] * 12, listed=[11, -1, 0, 7, 5, 12, 9, 2, -7, 4], V=60000), None, "full"),
    (dict(T=6, Hq=8, Hkv=1, cap=256, lens=[200] * 12, listed=[11, -1, 0, 7, 5, 12, 9, 2, -7, 4], V=60000), None, "slots"),
    (dict(T=30, Hq=16, Hkv=8, cap=700, lens=[700] * 12, listed=[11, -1, 0, 7, 5, 12, 9, 2, 1 << 30, 4], d=192, V=3001),
     None, "full"),
    (dict(T=61, Hq=64, Hkv=8, cap=4096, lens=[4000] * 4, listed=[3, -1, 1], d=192, V=3001, target=True), "splits", "full"),
    (dict(T=30, Hq=16, Hkv=8, cap=700, lens=[700] * 4, listed=[3, -1, 1, 4], d=192, V=3001), "pieces", "full"),
], ids=["beside", "gathered", "slots", "packed", "workspace", "pieces"])
def test_listed_sequences_that_do_not_exist_are_skipped_and_reported(kw, plan, room, monkeypatch):
    import torch
    from paper_2601_23180_b200 import binding as ts
    if plan:
        monkeypatch.setenv("TRISPEC_ATTN_PLAN", plan)
    good = Pass(**dict(kw, listed=[x for x in kw["listed"] if 0 <= x < len(kw["lens"])]))
    p = Pass(**kw)
    if plan:
        assert ts.trispec_verify_attn_plan(p.attn_args) == plan
    if room == "slots":
        p.lm_args.workspace_bytes -= len(kw["listed"]) * kw["T"] * 2048 * 2
    want = _want(good)
    for call in (p.separate, p.fused):
        p.spoil()
        p.status.zero_()
        call()
        p.snapshot(status=12)
        for b in range(p.B):
            if b not in p.seqs:                        # as spoil() left them
                assert torch.isnan(p.o[b].float()).all() and (p.stats["lse"][b] == 0).all()
                continue
            x, y = p.o[b].float(), p.attention64(b).float()
            # two bf16 steps of outputs of at most about 4, as in the parity tests
            assert (x - y).abs().max().item() <= 2e-2
            assert (p.stats["lse"][b] - good.stats["lse"][b]).abs().max().item() <= 1e-4
            assert torch.equal(p.stats["top1_idx"][b], want["s_top1_idx"][b])
            assert torch.equal(p.out["path"][b], want["d_path"][b])


@pytest.mark.parametrize("kw", [CHAINS, dict(T=61, Hq=16, Hkv=8, cap=4096, lens=[3000], paged=True)])
def test_stochastic_pass_beside(kw):
    import torch
    from paper_2601_23180_b200 import binding as ts
    p = Pass(**kw)
    g = torch.Generator(device="cuda")
    g.manual_seed(1)
    q = torch.rand(p.B, p.T, generator=g, device="cuda") * 1e-4 + 1e-6
    u = torch.rand(p.B, p.T, generator=g, device="cuda")
    p.scan_args = ts.scan_args(p.stats, p.parent, p.tok, 0.0, ts.MODE_PROXY, p.out, active=p.active, q_draft=q, u_accept=u)
    want = _want(p)
    for _ in range(3):
        p.spoil()
        p.fused()
        assert_same_attention(p.snapshot(), want)


@pytest.mark.parametrize("kw", [CHAINS, ONE, dict(T=61, Hq=16, Hkv=8, cap=4096, lens=[3000]),
                                dict(T=61, Hq=64, Hkv=8, cap=2048, lens=[1999], target=True)])
def test_malformed_tree_in_one_launch(kw):
    """A parent that comes later, in the last sequence: its node and all below it see nothing of the tree, and the status says so."""
    import torch
    p = Pass(**kw)
    p.parent[-1, 2] = 5
    want = None
    for call in (p.separate, p.fused, p.fused):
        p.spoil()
        p.status.zero_()
        n = launches(call)
        got = p.snapshot(status=11)
        if want is not None:
            assert want_n - n == ONE_LAUNCH
            assert_same_attention(got, want)
        want, want_n = want or got, n if want is None else want_n
    assert int(p.mask[-1, 2].item()) == 0 and int(p.depth[-1, 2].item()) == -1 and (p.mask[:, 0] == 1).all()


@pytest.mark.parametrize("kw", [
    dict(ONE, other_mask=True), dict(CHAINS, other_mask=True), dict(T=61, Hq=16, Hkv=8, cap=4096, lens=[3000], other_mask=True),
    dict(T=9, Hq=16, Hkv=8, cap=64, lens=[64] * 2048, listed=[5, 1999], V=32000),     # more trees than the launch takes along
])
def test_masks_of_a_launch_of_their_own(kw):
    import torch
    from paper_2601_23180_b200 import binding as ts
    kw = dict(kw)
    other = kw.pop("other_mask", False)
    p = Pass(**kw)
    if other:                                      # the attention follows chains, whatever the trees are
        chain = torch.tensor([(2 << i) - 1 for i in range(p.T)], dtype=torch.int64, device="cuda").repeat(p.B, 1).contiguous()
        p.attn_args.mask = chain.data_ptr()
    p.spoil()
    n = launches(p.separate)
    want = p.snapshot()
    for _ in range(3):
        p.spoil()
        assert n - launches(p.fused) == MASKS_APART
        assert_same_attention(p.snapshot(), want)
