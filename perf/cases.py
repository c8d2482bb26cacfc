"""What a decode loop asks of the library, as cases that can be timed and compared.

`call` says which public entry points one pass goes through:
  verify  trispec_verify with everything resident on the GPU: one verification of a batch of draft trees
  host    trispec_verify_host: the draft and its activations in pinned host memory, the decision read back
  sample  a round at temperature 1: trispec_verify with stochastic acceptance, trispec_sample_bonus for the
          sequences that need a sampled token, trispec_commit_kv of what was accepted
  target  the target's round for the sequences the proxy escalated: trispec_prune_tree at the last node the
          proxy accepted, then attention over the pruned trees, LM head, scan and trispec_commit_kv

The shapes are those of the package's configurations (`inputs.CONFIGS`) and of the paper's own setting
(one sequence), plus chains in a batch and an odd-sized batch. Inputs are drawn on the GPU from the seed:
activations, keys and values N(0, 1), weights N(0, 0.02^2), hidden states that favour a child's token with the
mixture of the package's input recipe, so that both routing cases occur.
"""
import math

import numpy as np
import torch

from paper_2601_23180_b200 import binding as ts
from paper_2601_23180_b200 import inputs as gen

D = 128


def _case(name, **over):
    c = dict(name=name, call="verify", B=1, active=0, k=60, tree="random", depth=6, L=4096, L_min=4096, Hq=16, Hkv=8,
             d=2048, V=151936, paged=False, target=False, entropy=False)
    c.update(over)
    return c


def listed():
    return [
        # one short request decoded alone with a chain draft: latency and launches are all there is
        _case("chain_1", k=8, tree="chain", depth=8, L=512, L_min=512, V=32000),
        # the paper's setting: one sequence, a tree of 60 drafts, verified by the proxy
        _case("tree_1", L=4096, L_min=4096),
        # the same sequence escalated: one full verification by the target
        _case("tree_1_target", L=8192, L_min=8192, Hq=64, d=5120, target=True),
        # a small batch of trees on the proxy
        _case("tree_8", B=8),
        # three of eight sequences were escalated and are verified by the target over long contexts
        _case("escalated_3_of_8", B=8, active=3, L=16384, L_min=16384, Hq=64, d=5120, target=True),
        # a medium batch with smaller, deeper trees and a wider model
        _case("tree_16", B=16, k=48, depth=8, L=8192, L_min=8192, Hq=32, d=4096, V=128256),
        # the largest: a serving batch of long, ragged reasoning contexts in a paged cache
        _case("tree_64_paged", B=64, L=32768, L_min=8192, paged=True),
        # a serving batch that drafts short chains instead of trees
        _case("chain_64_paged", B=64, k=8, tree="chain", depth=8, L=4096, L_min=512, Hq=32, d=4096, V=128256, paged=True),
        # the draft model runs elsewhere: inputs from host memory, the decision back on the host
        _case("tree_8_host", call="host", B=8),
        # a whole round at temperature 1, ragged batch, trees of 26 nodes
        _case("sampled_round_12", call="sample", B=12, k=25, depth=5, L=6000, L_min=700, Hq=32, d=4096, V=128256),
        # the target's round after the proxy accepted a prefix: pruned trees, then the commit
        _case("target_round_3_of_8", call="target", B=8, active=3, L=8192, L_min=2048, Hq=64, d=5120, paged=True,
              target=True),
        # odd sizes: five short sequences, 30 nodes, one query head per KV head, entropy routing, odd vocabulary
        _case("odd_5_entropy", B=5, k=29, depth=7, L=1777, L_min=130, Hq=16, Hkv=16, d=1024, V=50257, entropy=True),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """Batches of 1 to 64 sequences, chains of 2 to 10 drafts or trees of 12 to 63, contexts of 64 to 32768
    tokens, models from 1024 to 5120 wide with 1 to 8 query heads per KV head, vocabularies of 16000 to 152064."""
    while True:
        call = rng.choice(["verify"] * 6 + ["host", "sample", "target", "target"])
        B = _log(rng, 1, 64)
        chain = rng.random() < 0.35
        k = rng.randint(2, 10) if chain else rng.randint(12, 63)
        L = _log(rng, 64, 32768)
        L_min = L if rng.random() < 0.4 else rng.randint(max(1, L // 16), L)
        Hq, Hkv, d = rng.choice([(16, 8, 2048), (16, 8, 1024), (32, 8, 4096), (64, 8, 5120), (16, 16, 2048), (32, 8, 2560)])
        V = rng.choice([32000, 50257, 128256, 151936, rng.randint(16000, 152064), 8 * rng.randint(2000, 19008)])
        target = call == "target" or (call == "verify" and rng.random() < 0.3)
        active = 0
        if B > 1 and (call == "target" or (target and rng.random() < 0.6)):
            active = max(1, round(B * rng.uniform(0.1, 0.6)))
        c = _case("", call=call, B=B, active=active, k=k, tree="chain" if chain else "random",
                  depth=k if chain else rng.randint(3, 8), L=L, L_min=L_min, Hq=Hq, Hkv=Hkv, d=d, V=V,
                  paged=rng.random() < 0.5, target=target, entropy=(not target and rng.random() < 0.15))
        del c["name"]
        w, most = work(c), work(listed()[6])
        # no more work than the largest listed case, and its inputs fit on the card several times over
        room = 3e9 if call in ("sample", "target") else 12e9
        if w["flops"] <= most["flops"] and w["bytes"] <= most["bytes"] and 2 * B * L * Hkv * D * 2 <= room:
            return c


def _n_active(c):
    return c["active"] or c["B"]


def _mean_nodes(c):
    """Tree nodes of a sequence that the pass has to look at (about half of them remain after pruning)."""
    T = c["k"] + 1
    return (T + 1) / 2 if c["call"] == "target" else T


def work(c):
    n, T = _n_active(c), _mean_nodes(c)
    ctx = n * (c["L"] + c["L_min"]) / 2
    rows = n * T
    kv = 2 * (ctx + rows) * c["Hkv"] * D * 2
    qo = 2 * rows * c["Hq"] * D * 2
    lm = c["V"] * c["d"] * 2 + rows * c["d"] * 2
    small = n * (c["k"] + 1) * 76
    flops = 4 * c["Hq"] * D * T * (ctx + rows) + 2 * rows * c["d"] * c["V"]
    return {"bytes": kv + qo + lm + small, "flops": flops}


def tolerance(c):
    # The widest outputs are the attention's: bf16, from probabilities rounded to bf16 (relative errors of up to
    # 2^-9 each). Against 64-bit arithmetic on the same inputs they are off by 2.3e-3 to 2.9e-3 in the 2-norm and by
    # at most 1.8e-2 of the root mean square in one value (the statistics by 2e-5 and 4e-5); four times that is
    # allowed. Whole numbers differ where two logits tie in 32 bits.
    return {"rel": 1.2e-2, "max": 7e-2, "differ": 2e-3}

def _ragged(rng, c):
    if c["L_min"] >= c["L"]:
        return np.full(c["B"], c["L"], dtype=np.int32)
    return rng.integers(c["L_min"], c["L"] + 1, size=c["B"]).astype(np.int32)


def prepare(case, seed):
    c = case
    B, T, d, V, Hq, Hkv = c["B"], c["k"] + 1, c["d"], c["V"], c["Hq"], c["Hkv"]
    dev = "cuda"
    rng = np.random.default_rng([seed & 0x7FFFFFFF, 17])
    g = torch.Generator(device=dev)
    g.manual_seed(seed)

    def normal(*shape, std=1.0):
        x = torch.randn(*shape, generator=g, device=dev, dtype=torch.bfloat16)
        return x if std == 1.0 else x.mul_(std)

    def i32(a):
        return torch.from_numpy(np.ascontiguousarray(a, dtype=np.int32)).to(dev)

    # ---- draft trees and tokens
    cfg = gen.VerifyConfig("case", B=B, k=c["k"], tree=c["tree"], max_depth=c["depth"], L=c["L"], Hq=Hq, Hkv=Hkv, d=d, V=V,
                           logit_scale=1.0, seed=seed)
    parent_np = np.stack([gen.make_tree(cfg, b) for b in range(B)])
    tok_np = np.stack([gen.make_tokens(cfg, b, parent_np[b]) for b in range(B)])

    # ---- LM head weights and hidden states that favour one child's token (confidently in 70 % of the nodes)
    W = normal(V, d, std=0.02)
    fav = rng.integers(0, V, size=(B, T))
    order = rng.permutation(T - 1) + 1
    rows = np.arange(B)
    for n in order:                                   # the last child written is the favoured one
        fav[rows, parent_np[:, n]] = tok_np[:, n]
    alpha = np.where(rng.random((B, T)) < 0.7, 8.0, 1.0).astype(np.float32)
    w = W[torch.from_numpy(fav.reshape(-1)).to(dev)].float()
    w = w / w.norm(dim=1, keepdim=True) * torch.from_numpy(alpha.reshape(-1, 1)).to(dev)
    h = (w + torch.randn(w.shape, generator=g, device=dev)).to(torch.bfloat16).view(B, T, d)
    logit_scale = 3.6 / (0.02 * math.sqrt(d))

    # ---- attention inputs and the KV cache
    q, kt, vt = normal(B, T, Hq, D), normal(B, T, Hkv, D), normal(B, T, Hkv, D)
    ctx_np = _ragged(rng, c)
    grows = c["call"] in ("sample", "target")         # room for the rows that a round appends
    room = T if grows else 0
    table = None
    if c["paged"]:
        need = (ctx_np.astype(np.int64) + room + 63) // 64
        per_seq = (c["L"] + room + 63) // 64          # the pool holds every sequence at its longest
        perm = rng.permutation(B * per_seq).astype(np.int32)
        table_np = np.full((B, per_seq), -1, dtype=np.int32)
        at = 0
        for b in range(B):
            table_np[b, :need[b]] = perm[at:at + need[b]]
            at += int(need[b])
        table = i32(table_np)
        kc, vc = normal(B * per_seq, 64, Hkv, D), normal(B * per_seq, 64, Hkv, D)
    else:
        kc, vc = normal(B, c["L"] + room, Hkv, D), normal(B, c["L"] + room, Hkv, D)
    ctx = i32(ctx_np)

    # ---- which sequences take part
    seq_index, active = None, torch.ones(B, dtype=torch.uint8, device=dev)
    if c["active"]:
        chosen = np.sort(rng.permutation(B)[:c["active"]]).astype(np.int32)
        seq_index = i32(chosen)
        active.zero_()
        active[torch.from_numpy(chosen.astype(np.int64)).to(dev)] = 1

    s = dict(case=c, keep=(W, q, kt, vt, kc, vc, h))
    if c["call"] == "host":
        # per-round arrays in pinned host memory, each group back to back like its copy on the GPU
        i, b16 = torch.int32, torch.bfloat16
        flats = []
        host, there = {}, {}
        for group in ([("parent", parent_np), ("tok", tok_np), ("h", h)], [("q", q), ("k_tree", kt), ("v_tree", vt)]):
            specs = [(n, tuple(a.shape), i if isinstance(a, np.ndarray) else b16) for n, a in group]
            flat = torch.zeros(ts._carve_bytes(specs), dtype=torch.uint8).pin_memory()
            for n, view in ts._carve(flat, specs).items():
                a = dict(group)[n]
                view.copy_(torch.from_numpy(a) if isinstance(a, np.ndarray) else a)
                host[n] = view
            copy = torch.zeros(flat.numel(), dtype=torch.uint8, device=dev)
            there.update(ts._carve(copy, specs))
            flats += [flat, copy]
        parent, tok, h, q, kt, vt = (there[n] for n in ("parent", "tok", "h", "q", "k_tree", "v_tree"))
        specs = ts.scan_out_specs(B, T)
        back = torch.zeros(ts._carve_bytes(specs), dtype=torch.uint8).pin_memory()
        host.update(ts._carve(back, specs))
        s["host"], s["io"], s["flats"] = host, ts.host_io(**host), (flats, back)
    else:
        parent, tok = i32(parent_np), i32(tok_np)

    status = torch.zeros(1, dtype=torch.int32, device=dev)
    mask = torch.zeros((B, T), dtype=torch.int64, device=dev)
    depth = torch.zeros((B, T), dtype=torch.int32, device=dev)
    stats = ts.alloc_stats(B, T, entropy=c["entropy"])
    scan_out = ts.alloc_scan_out(B, T)
    o = torch.zeros((B, T, Hq, D), dtype=torch.bfloat16, device=dev)
    lse = torch.zeros((B, Hq, T), dtype=torch.float32, device=dev)
    n_nodes = None
    if c["call"] == "target":
        # the proxy's pass left the full tree's mask and, per sequence, the last node it accepted: the root for
        # most sequences (nothing was trusted), one of the root's children or grandchildren for the others
        s["tree"] = ts.tree_args(parent, mask, depth, dev_status=status)
        ts.trispec_build_tree_mask(s["tree"])
        root_np = np.full(B, -1, dtype=np.int32)
        for b in (np.arange(B) if seq_index is None else chosen):
            r = 0
            for _ in range(int(rng.integers(0, 3))):
                kids = np.nonzero(parent_np[b] == r)[0]
                if len(kids):
                    r = int(rng.choice(kids))
            root_np[b] = r
        out = ts.alloc_prune_out(B, T)
        s["prune"], s["pruned"] = ts.prune_args(parent, tok, mask, i32(root_np), out), out
        parent, tok, mask, n_nodes = out["parent"], out["tok"], out["mask"], out["n_keep"]
    else:
        s["tree"] = ts.tree_args(parent, mask, depth, dev_status=status)
    a = ts.attn_args(q, kt, vt, mask, kc, vc, ctx, 1.0 / math.sqrt(D), o, block_table=table, seq_index=seq_index, lse=lse,
                     dev_status=status, n_nodes=n_nodes)
    ws_a = ts.alloc_workspace(ts.trispec_verify_attn_workspace(a))
    a.workspace, a.workspace_bytes = ws_a.data_ptr(), ws_a.numel()
    l = ts.lmhead_args(h, W, parent, tok, logit_scale, stats, seq_index=seq_index, dev_status=status)
    ws_l = ts.alloc_workspace(ts.trispec_lmhead_stats_workspace(l))
    l.workspace, l.workspace_bytes = ws_l.data_ptr(), ws_l.numel()
    more = {}
    if c["call"] == "sample":
        more = dict(q_draft=torch.rand(B, T, generator=g, device=dev) * 0.95 + 0.05,
                    u_accept=torch.rand(B, T, generator=g, device=dev))
    s["scan"] = ts.scan_args(stats, parent, tok, 1.2 if c["entropy"] else 0.5, ts.MODE_TARGET if c["target"] else ts.MODE_PROXY,
                             scan_out, active=active, criterion=ts.CRIT_ENTROPY if c["entropy"] else ts.CRIT_MARGIN, **more)
    s["attn"], s["lm"], s["ws"] = a, l, (ws_a, ws_l)
    s["out"] = dict(o=o, attn_lse=lse, stats=stats, scan=scan_out, status=status)
    if c["call"] == "target":
        s["out"]["pruned"] = out
    else:
        s["out"].update(mask=mask, depth=depth)
    if c["call"] == "sample":
        value = torch.zeros(B, dtype=torch.float32, device=dev)
        b = ts.sample_args(h, W, scan_out["last_node"], scan_out["bonus_tok"], logit_scale, seed, 7, sample_value=value,
                           dev_status=status)
        ws_b = ts.alloc_workspace(ts.trispec_sample_bonus_workspace(b))
        b.workspace, b.workspace_bytes = ws_b.data_ptr(), ws_b.numel()
        s["bonus"], s["ws"] = b, (ws_a, ws_l, ws_b)
        s["out"]["sample_value"] = value
    if grows:
        # the new lengths go to the other of two arrays, as in a loop that keeps the last round's
        ctx_out = torch.zeros(B, dtype=torch.int32, device=dev)
        s["commit"] = ts.commit_args(kt, vt, kc, vc, ctx, scan_out["path"], scan_out["accept_len"], ctx_out,
                                     block_table=table, active=active, dev_status=status)
        s["out"].update(ctx_len=ctx_out, k_cache=kc, v_cache=vc)
    return s


def run(s):
    call = s["case"]["call"]
    if call == "host":
        ts.trispec_verify_host(s["io"], s["tree"], s["attn"], s["lm"], s["scan"])
        torch.cuda.current_stream().synchronize()     # the loop reads the decision on the host
        return dict(s["out"], host={n: s["host"][n] for n, _, _ in ts.scan_out_specs(1, 1)})
    if call == "target":
        ts.trispec_prune_tree(s["prune"])
        ts.trispec_verify_attn(s["attn"])
        ts.trispec_lmhead_stats(s["lm"])
        ts.trispec_accept_scan(s["scan"])
    else:
        ts.trispec_verify(s["tree"], s["attn"], s["lm"], s["scan"])
    if call == "sample":
        ts.trispec_sample_bonus(s["bonus"])
    if "commit" in s:
        ts.trispec_commit_kv(s["commit"])
    return s["out"]
