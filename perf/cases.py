"""What a user of this library waits for: single queries, batches, host results, compact results, the
per-snapshot recompute, and loading a graph, from a few thousand vertices to four million.

Every case is an evolving RMAT graph (``V`` vertices, ``E`` edges in the first snapshot, ``S`` snapshots,
``step`` deletions and as many additions between two snapshots, weights uniform in [1, 999]) and one call on
it.  The graph is the handle a program keeps: it is drawn from the case alone, loaded once and kept; the
sources and windows of a state's queries come from the seed.  Only the load case draws its graph from the
seed, since there the graph is the input.
"""
from __future__ import annotations

import math
from collections import OrderedDict
from types import SimpleNamespace

import numpy as np
import torch

from paper_2502_10579_gb300 import svv

SSSP, SSWP, BFS, SSNP = svv.SVV_SSSP, svv.SVV_SSWP, svv.SVV_BFS, svv.SVV_SSNP
INF = 0xFFFFFFFF
MIXED = -1   # a batch: a third each of SSSP, SSWP and BFS
KEPT = 6     # graphs a process keeps loaded


def listed():
    small = dict(V=4096, E=32768, S=8, step=328)
    g64k = dict(V=1 << 16, E=1 << 20, S=64, step=262)
    g1m = dict(V=1 << 20, E=1 << 24, S=64, step=10000)
    g4m = dict(V=1 << 22, E=1 << 26, S=64, step=16777)
    return [
        # the smallest graph in use (the configuration of the smoke test): one query, where launches and rounds count
        dict(name="query_4k", call="query", type=SSSP, win_len=8, n=1, **small),
        # an interactive query on a small graph: hop counts over a short recent window
        dict(name="query_64k_bfs", call="query", type=BFS, win_len=16, n=1, **g64k),
        # many users' queries on a small graph in one call (the batch mix: types, sources, windows of 8 to 64)
        dict(name="batch_64k", call="batch", type=MIXED, win_len=0, n=64, **g64k),
        # odd sizes and two mask words per edge: a minimax-path query over 77 of 100 snapshots
        dict(name="query_300k_odd", call="query", type=SSNP, win_len=77, n=1, V=300007, E=4700001, S=100, step=4700),
        # the benchmark's graph: shortest paths over its whole history
        dict(name="query_1m_sssp", call="query", type=SSSP, win_len=64, n=1, **g1m),
        # the same graph, widest paths over a short window somewhere in the history
        dict(name="query_1m_window", call="query", type=SSWP, win_len=8, n=1, **g1m),
        # the benchmark's step: SSSP and SSWP of one source over one window, as one mixed group
        dict(name="pair_1m", call="pair", type=MIXED, win_len=64, n=2, **g1m),
        # results a program reads on the host, written to page-locked memory
        dict(name="host_1m", call="host", type=BFS, win_len=32, n=1, **g1m),
        # only the rows that change: what a program stores or sends on
        dict(name="compact_1m", call="compact", type=SSSP, win_len=32, n=1, **g1m),
        # the plain recompute, for callers that want a few separate snapshots
        dict(name="plain_1m", call="plain", type=SSWP, win_len=8, n=1, **g1m),
        # the largest: a batch on a graph of four million vertices, in query groups
        dict(name="batch_4m", call="batch", type=MIXED, win_len=0, n=16, **g4m),
        # a new edge log arrives: build the versioned graph, load it, answer the first query
        dict(name="load_256k", call="load", type=SSSP, win_len=16, n=1, V=1 << 18, E=1 << 22, S=64, step=1049),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choice(["query", "query", "query", "batch", "pair", "host", "compact", "plain", "load"])
    top = {"load": 1 << 18, "plain": 1 << 20, "batch": 1 << 22}.get(call, 1 << 21)
    V = min(top, max(4096, _log_uniform(rng, 4096, top) | rng.randint(0, 1)))
    E = V * rng.randint(4, 15) + rng.randint(0, V)
    S = rng.choice([8, 32, 64, 100, 128, rng.randint(2, 128)])
    step = max(1, int(E * math.exp(rng.uniform(math.log(0.0002), math.log(0.005)))))
    if V > 1 << 20:
        step = min(step, E // 1000)
    L = rng.randint(1, S)
    if call == "plain":
        L = min(L, 8)
    if call == "batch":
        return dict(call=call, type=MIXED, win_len=0, n=rng.randint(3, 16 if V > 1 << 18 else 64), V=V, E=E, S=S, step=step)
    if call == "pair":
        return dict(call=call, type=MIXED, win_len=L, n=2, V=V, E=E, S=S, step=step)
    return dict(call=call, type=rng.choice([SSSP, SSWP, BFS, SSNP]), win_len=L, n=1, V=V, E=E, S=S, step=step)


# ---- inputs ------------------------------------------------------------------

def _rmat(gen, V, n):
    """n RMAT (0.57, 0.19, 0.19, 0.05) endpoint pairs, scaled onto V vertices."""
    levels = max(1, (V - 1).bit_length())
    src = torch.zeros(n, dtype=torch.int64, device="cuda")
    dst = torch.zeros(n, dtype=torch.int64, device="cuda")
    for _ in range(levels):
        r = torch.rand(n, generator=gen, device="cuda")
        row = r >= 0.76
        col = ((r >= 0.57) & ~row) | (r >= 0.95)
        src.mul_(2).add_(row)
        dst.mul_(2).add_(col)
    return ((src * V) >> levels).to(torch.int32), ((dst * V) >> levels).to(torch.int32)


def _log(case, seed):
    """The evolving graph as edge instances: (src, dst, weight, added in step, deleted in step)."""
    V, E, S = case["V"], case["E"], case["S"]
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    src, dst = _rmat(gen, V, E)
    srcs, dsts, adds, dels = [src], [dst], [torch.zeros(E, dtype=torch.int32, device="cuda")], []
    live = torch.arange(E, dtype=torch.int64, device="cuda")
    total = E
    for s in range(1, S):
        pos = torch.randint(0, E, (case["step"],), generator=gen, device="cuda").unique()
        k = pos.shape[0]
        dels.append((live[pos], s))
        u, v = _rmat(gen, V, k)
        srcs.append(u)
        dsts.append(v)
        adds.append(torch.full((k,), s, dtype=torch.int32, device="cuda"))
        live[pos] = torch.arange(total, total + k, device="cuda")
        total += k
    t_del = torch.full((total,), S, dtype=torch.int32, device="cuda")
    for ids, s in dels:
        t_del[ids] = s
    w = torch.randint(1, 1000, (total,), generator=gen, device="cuda", dtype=torch.int32)
    return torch.cat(srcs), torch.cat(dsts), w, torch.cat(adds), t_del


def _csr(case, log):
    """The log as the versioned CSR of svv_load, on the device."""
    V, S = case["V"], case["S"]
    src, dst, w, t_add, t_del = log
    order = torch.sort(src, stable=True).indices
    row_ptr = torch.zeros(V + 1, dtype=torch.int64, device="cuda")
    row_ptr[1:] = torch.bincount(src, minlength=V).cumsum(0)

    def below(t):  # bits 0..t-1
        return torch.where(t >= 64, torch.full_like(t, -1), (torch.ones_like(t) << t.clamp(max=63)) - 1)

    a, d = t_add[order].long(), t_del[order].long()
    words = [below((d - 64 * j).clamp(0, 64)) & ~below((a - 64 * j).clamp(0, 64)) for j in range((S + 63) // 64)]
    return row_ptr, dst[order].contiguous(), w[order].contiguous(), torch.stack(words, 1).contiguous()


_graphs: OrderedDict = OrderedDict()


def _graph(case):
    """(context with the case's graph loaded, vertices with an out-edge in the first snapshot)."""
    pair = case["call"] == "pair"
    key = (case["V"], case["E"], case["S"], case["step"], pair)
    if key not in _graphs:
        while len(_graphs) >= KEPT:
            _graphs.popitem(last=False)
        log = _log(case, 1000 + case["S"])
        ctx = svv.Context(0)
        if pair:
            ctx.set_tuning("batch_mode", 2)
            ctx.set_tuning("group_mix", 1)
        csr = _csr(case, log)
        torch.cuda.synchronize()
        ctx.load_csr(case["V"], case["S"], *csr, inputs_on_device=True)
        used = torch.bincount(log[0][:case["E"]], minlength=case["V"]).nonzero().flatten().cpu().numpy()
        del log, csr
        torch.cuda.empty_cache()
        _graphs[key] = (ctx, used)
    _graphs.move_to_end(key)
    return _graphs[key]


def _lengths(case):
    """Window lengths of a batch: 8 to 64 snapshots, the same for every seed so that results keep their shapes."""
    hi = min(64, case["S"])
    return np.random.default_rng(case["n"]).integers(min(8, hi), hi + 1, size=case["n"]).tolist()


def _queries(case, seed, used):
    """[(type, source, first snapshot, length)] of a state."""
    rng = np.random.default_rng(seed)
    V, S, n = case["V"], case["S"], case["n"]

    def window(L):
        return int(rng.integers(0, S - L + 1)), L

    if case["call"] == "batch":  # uniform sources, types in shuffled order
        kinds = rng.permutation(np.resize([SSSP, SSWP, BFS], n)).tolist()
        return [(t, int(rng.integers(0, V)), *window(L)) for t, L in zip(kinds, _lengths(case))]
    source, win = int(rng.choice(used)), window(case["win_len"])
    types = [SSSP, SSWP] if case["call"] == "pair" else [case["type"]]
    return [(t, source, *win) for t in types]


def prepare(case, seed):
    call, V = case["call"], case["V"]
    st = SimpleNamespace(call=call, log=None)
    if call == "load":
        log = _log(case, seed)
        used = torch.bincount(log[0][:case["E"]], minlength=V).nonzero().flatten().cpu().numpy()
        names = ("src", "dst", "w", "t_add", "t_del")
        st.log = SimpleNamespace(V=V, S=case["S"], **{k: x.cpu().numpy().view(np.uint32) for k, x in zip(names, log)})
        st.ctx = svv.Context(0)
    else:
        st.ctx, used = _graph(case)
    st.queries = _queries(case, seed, used)
    if call == "host":
        st.outs = [torch.zeros((q[3], V), dtype=torch.int32).pin_memory() for q in st.queries]
    else:
        st.outs = [torch.zeros((q[3], V), dtype=torch.int32, device="cuda") for q in st.queries]
    if call == "compact":
        st.cap, st.row = (torch.zeros(V, dtype=torch.int32, device="cuda") for _ in range(2))
    return st


def run(st):
    q = st.queries[0]
    if st.call in ("batch", "pair"):
        outs, _ = st.ctx.query_batch([(*p, out) for p, out in zip(st.queries, st.outs)])
        return outs
    if st.call == "host":
        return st.ctx.query_host(*q, st.outs[0])
    if st.call == "plain":
        return st.ctx.query(*q, out=st.outs[0], plain=True)
    if st.call == "compact":
        rows = svv.svv_query_compact(st.ctx.h, *q, st.cap, st.row, st.outs[0])
        return {"rows": rows, "cap": st.cap, "row": st.row, "values": st.outs[0]}
    if st.call == "load":
        st.ctx.load_log(st.log)
    return st.ctx.query(*q, out=st.outs[0])


def work(case):
    """The graph once (offsets, targets, weights, the masks of the edges that come or go), each result once."""
    V, S, words = case["V"], case["S"], (case["S"] + 63) // 64
    inst = case["E"] + (S - 1) * case["step"]
    partial = min(inst, 2 * (S - 1) * case["step"])
    graph = 4 * V + (4 if case["type"] == BFS else 8) * inst + 8 * words * partial
    lengths = _lengths(case) if case["call"] == "batch" else [case["win_len"]] * case["n"]
    out = 4 * V * sum(lengths)
    if case["call"] == "load":
        graph += 20 * inst  # the log
    return {"bytes": graph + out, "flops": inst * case["n"]}


# ---- the same results from the definition -------------------------------------

def _solve(V, t, source, src, dst, w):
    """Values of every vertex by rounds of relaxing every edge, in 64 bits."""
    wide = t == SSWP
    val = torch.full((V,), 0 if wide else INF, dtype=torch.int64, device="cuda")
    val[source] = INF if wide else 0
    while True:
        v = val[src]
        if t == SSSP:
            cand = torch.where(v == INF, v, (v + w).clamp(max=INF - 1))
        elif t == BFS:
            cand = torch.where(v == INF, v, v + 1)
        else:
            cand = torch.minimum(v, w) if wide else torch.maximum(v, w)
        new = val.scatter_reduce(0, dst, cand, "amax" if wide else "amin")
        if torch.equal(new, val):
            return val
        val = new


def exact(case, seed):
    inst = case["E"] + (case["S"] - 1) * case["step"]
    total = sum(_lengths(case)) if case["call"] == "batch" else case["win_len"] * case["n"]
    if inst * total > 2.5e9:
        return None  # over 20 seconds
    log = _log(case, seed if case["call"] == "load" else 1000 + case["S"])
    used = torch.bincount(log[0][:case["E"]], minlength=case["V"]).nonzero().flatten().cpu().numpy()
    src, dst, w, t_add, t_del = (x.long() for x in log)

    def signed(x):  # as the 32-bit words of the results read
        return torch.where(x > 0x7FFFFFFF, x - (1 << 32), x)

    def graph(keep):
        return src[keep], dst[keep], w[keep]

    outs = []
    for t, source, b, L in _queries(case, seed, used):
        if case["call"] == "compact":
            cap = _solve(case["V"], t, source, *graph((t_add <= b) & (t_del >= b + L)))
            cup = _solve(case["V"], t, source, *graph((t_add < b + L) & (t_del > b)))
            return {"rows": int((cap != cup).sum()), "cap": signed(cap), "row": None, "values": None}
        rows = [signed(_solve(case["V"], t, source, *graph((t_add <= i) & (t_del > i)))) for i in range(b, b + L)]
        outs.append(torch.stack(rows))
    return outs if case["call"] in ("batch", "pair") else outs[0]
