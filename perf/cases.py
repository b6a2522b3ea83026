"""Performance cases of the engine: what a program that tracks Random Walk with
Restart scores on a changing graph asks of it, through the public entry points.

A case is a dict of plain values:

  kind    "update": apply a batch of updates, read every tracked score vector,
          apply the batch that takes the changes back (edges that expire, nodes
          that leave), read the vectors again. "cpi": scores from scratch and
          one read. "topk": the k best nodes of up to 32 tracked seeds.
  graph   "er" (uniform), "rmat" (power law, directed) or "chunglu" (power
          law, undirected, stored both ways); n nodes and at most m edges
          (pairs for "chunglu").
  seeds   tracked seeds (one: the one-seed path; more: the seed block).
  prec    "f64", "f32" or "bf16": the engine's precision. Scores of the two
          mixed precisions are handed on as float32, those of "f64" as float64.
  ops     edge operations of a batch (pairs for "chunglu"), half insertions of
          absent edges, half deletions of present ones.
  nodes   nodes a batch adds, each with out-edges and in-edges; the batch that
          takes the changes back deletes them.
  eps     the stopping tolerance of the updates; the initial scores are taken
          to a hundredth of it.
  order, graphs, det, device: engine options (node order, CUDA graphs,
          deterministic mode) and the form of the batch (in device memory or a
          host array).

Everything is drawn from the seed given to ``prepare``.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1712_00595_gb300 import native as N

C = 0.15  # restart probability of every case
PREC = {"f64": N.OSP_PREC_FP64, "f32": N.OSP_PREC_FP32_ACC64, "bf16": N.OSP_PREC_BF16_ACC64}
OUT_EDGES, IN_EDGES = 8, 8  # of every added node


def _case(kind, graph, n, m, **kw):
    c = dict(kind=kind, graph=graph, n=n, m=m, seeds=1, prec="f32", ops=0, nodes=0, eps=1e-6, k=0,
             order=0, graphs=False, device=False, det=False)
    c.update(kw)
    return c


def listed():
    """The work of this engine's users, from the smallest calls to the largest."""
    named = [
        # exact scores on a small graph, batch by batch: many short steps, where latency counts
        ("er10k_exact_f64", _case("update", "er", 10_000, 100_000, prec="f64", ops=100, eps=1e-12)),
        # one edge comes or goes and the scores follow at once (odd node count, CUDA graphs)
        ("one_edge_f32", _case("update", "rmat", 100_003, 1_200_000, ops=1, graphs=True)),
        # one seed on a large power-law graph, a batch of 1,000 already on the device
        ("rmat20_f32", _case("update", "rmat", 1 << 20, 1 << 24, ops=1000, graphs=True,
                             device=True)),
        # double precision throughout, odd sizes, a batch near the limit of one unit
        ("odd_f64_10k_ops", _case("update", "rmat", 300_007, 3_000_017, prec="f64", ops=10_001,
                                  eps=1e-9)),
        # an import: one host batch of 60,000 operations, more than one unit
        ("bulk_f32_60k_ops", _case("update", "rmat", 1 << 18, 1 << 22, ops=60_000, eps=1e-8)),
        # scores from scratch, the start of every program (and the static baseline)
        ("cpi_f32", _case("cpi", "rmat", 1 << 19, 1 << 23, eps=1e-6)),
        # 64 users of an undirected social graph
        ("chunglu_s64_f32", _case("update", "chunglu", 1 << 18, 1 << 21, seeds=64, ops=500,
                                  order=1)),
        # a few seeds in double precision, odd sizes
        ("block17_f64", _case("update", "rmat", 65_537, 1_000_003, seeds=17, prec="f64", ops=333,
                              eps=1e-9)),
        # a middling bf16 block with a partly filled last column group and a small batch
        ("block100_bf16", _case("update", "rmat", 131_071, 1_500_000, seeds=100, prec="bf16",
                                ops=200, order=1)),
        # the benchmark's 256-seed block (nodes come and go) at a size that loads quickly
        ("nodes_s256_bf16", _case("update", "rmat", 1 << 21, 1 << 25, seeds=256, prec="bf16",
                                  ops=500, nodes=500, order=1)),
        # 256 seeds from scratch (float rows, as for every bf16 block's start)
        ("cpi_s256_bf16", _case("cpi", "rmat", 1 << 18, 1 << 22, seeds=256, prec="bf16", eps=1e-4,
                                order=1)),
        # serving: the best 100 nodes of 32 tracked seeds as one query
        ("topk32", _case("topk", "rmat", 1 << 21, 1 << 24, seeds=64, prec="f64", k=100, eps=1e-4)),
    ]
    return [dict(c, name=name) for name, c in named]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges."""
    kind = rng.choice(["one", "one", "block", "block", "cpi", "topk"])
    deg = rng.choice([8, 12, 16])
    if kind == "one":
        n = _log(rng, 5_000, 600_000)
        prec = rng.choice(["f64", "f32"])
        return _case("update", rng.choice(["er", "rmat", "chunglu"]), n, n * deg // 2, prec=prec,
                     ops=_log(rng, 1, max(2, min(30_000, n // 8))),
                     nodes=rng.choice([0, 0, _log(rng, 1, 300)]),
                     eps=rng.choice([1e-4, 1e-6, 1e-8] + ([1e-10] if prec == "f64" else [])),
                     order=rng.choice([0, 1]), graphs=rng.choice([True, False]),
                     device=rng.choice([True, False]), det=rng.random() < 0.2)
    if kind == "block":
        n = _log(rng, 5_000, 200_000)
        return _case("update", rng.choice(["rmat", "chunglu"]), n, n * deg // 2,
                     seeds=_log(rng, 2, 256), prec=rng.choice(["f64", "f32", "bf16", "bf16"]),
                     ops=_log(rng, 1, max(2, min(5_000, n // 8))),
                     nodes=rng.choice([0, 0, _log(rng, 1, 300)]),
                     eps=rng.choice([1e-4, 1e-6, 1e-8]), order=rng.choice([0, 1, 1]),
                     graphs=rng.choice([True, False]))
    if kind == "cpi":
        many = rng.random() < 0.5
        n = _log(rng, 5_000, 100_000 if many else 400_000)
        return _case("cpi", "rmat", n, n * deg, seeds=_log(rng, 2, 256) if many else 1,
                     prec=rng.choice(["f64", "f32"]), eps=rng.choice([1e-4, 1e-6, 1e-8]),
                     order=rng.choice([0, 1]))
    n = _log(rng, 10_000, 600_000)
    return _case("topk", "rmat", n, n * deg, seeds=rng.choice([1, _log(rng, 2, 64)]), prec="f64",
                 k=rng.choice([1, 10, 100, 128]), eps=1e-4, order=rng.choice([0, 1]))


# --------------------------------------------------------------------------
# Inputs
# --------------------------------------------------------------------------
class _Sampler:
    """Random (u, v) pairs of one graph model, as keys (u << 32) | v on the GPU."""

    def __init__(self, case, gen):
        self.kind, self.n, self.gen = case["graph"], case["n"], gen
        self.levels = max(1, (self.n - 1).bit_length())
        if self.kind == "rmat":
            self.perm = torch.randperm(1 << self.levels, generator=gen, device="cuda")
        elif self.kind == "chunglu":
            w = torch.arange(1, self.n + 1, dtype=torch.float64, device="cuda") ** (-1.0 / 1.1)
            w *= 16.0 * self.n / w.sum()
            w.clamp_(max=float(w.sum().sqrt()))
            self.cdf = torch.cumsum(w / w.sum(), 0)
            self.perm = torch.randperm(self.n, generator=gen, device="cuda")

    def _rand(self, k):
        return torch.rand(k, generator=self.gen, device="cuda")

    def pairs(self, k):
        """About k pairs without self-loops (for "chunglu" the smaller id first)."""
        if self.kind == "rmat":
            u = torch.zeros(k, dtype=torch.int64, device="cuda")
            v = torch.zeros_like(u)
            for _ in range(self.levels):  # quadrants (.57, .19, .19, .05)
                r = self._rand(k)
                u = (u << 1) | (r >= 0.76)
                v = (v << 1) | (((r >= 0.57) & (r < 0.76)) | (r >= 0.95))
            u, v = self.perm[u], self.perm[v]
        elif self.kind == "chunglu":
            d = torch.rand(2, k, generator=self.gen, device="cuda", dtype=torch.float64)
            u, v = self.perm[torch.searchsorted(self.cdf, d).clamp_(max=self.n - 1)]
            u, v = torch.minimum(u, v), torch.maximum(u, v)
        else:
            u, v = torch.randint(0, self.n, (2, k), generator=self.gen, device="cuda")
        ok = (u != v) & (u < self.n) & (v < self.n)
        return (u[ok] << 32) | v[ok]

    def graph(self, m):
        """At most m distinct keys, ascending."""
        share = (self.n / (1 << self.levels)) ** 2 if self.kind == "rmat" else 1.0
        keys = torch.unique(self.pairs(int(1.15 * m / share) + 64))
        if keys.numel() > m:
            pick = torch.randperm(keys.numel(), generator=self.gen, device="cuda")[:m]
            keys = keys[pick].sort().values
        return keys

    def absent(self, keys, k):
        """k distinct pairs that are not in the ascending ``keys``."""
        got = torch.empty(0, dtype=torch.int64, device="cuda")
        while got.numel() < k:
            cand = torch.cat([got, self.pairs(4 * k + 64)])
            at = torch.searchsorted(keys, cand).clamp_(max=keys.numel() - 1)
            got = torch.unique(cand[keys[at] != cand])
        return got[torch.randperm(got.numel(), generator=self.gen, device="cuda")[:k]]


def _split(keys):
    return keys >> 32, keys & 0xFFFFFFFF


def _both(keys):
    """Every pair in both directions."""
    u, v = _split(keys)
    return torch.cat([keys, (v << 32) | u])


def _rows(keys, op):
    u, v = _split(keys)
    return torch.stack([u, v, torch.full_like(u, op)], 1)


def _draw_inputs(case, seed):
    """Graph, seeds and the two batches of a case. Ids from n on name the nodes
    that a pass adds."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    n, ops, nodes = case["n"], case["ops"], case["nodes"]
    both = case["graph"] == "chunglu"
    smp = _Sampler(case, gen)

    def perm(k):
        return torch.randperm(k, generator=gen, device="cuda")

    keys = smp.graph(case["m"])
    edges = _both(keys) if both else keys
    deg = torch.bincount(edges >> 32, minlength=n)
    # tracked seeds: the nodes of highest out-degree for one seed and for rankings
    # (whose order must not hang on ties), else uniform over the nodes
    if case["seeds"] == 1 or case["kind"] == "topk":
        seeds = torch.argsort(deg, descending=True, stable=True)[: case["seeds"]]
    else:
        seeds = perm(n)[: case["seeds"]]
    there = back = None
    if case["kind"] == "update":
        n_ins = (ops + 1) // 2
        ins = smp.absent(keys, n_ins)
        gone = keys[perm(keys.numel())[: ops - n_ins]]
        if both:
            ins, gone = _both(ins), _both(gone)
        edit = torch.cat([_rows(ins, 0), _rows(gone, 1)])
        undo = torch.cat([_rows(ins, 1), _rows(gone, 0)])
        edit, undo = edit[perm(edit.shape[0])], undo[perm(undo.shape[0])]
        if nodes:
            new = torch.arange(n, n + nodes, device="cuda")
            zero = torch.zeros_like(new)
            add = torch.stack([zero, zero, torch.full_like(new, 2)], 1)
            # in-edges come from the sources of random edges (busy nodes more often)
            src = edges[torch.randint(0, edges.numel(), (nodes * IN_EDGES,), generator=gen,
                                      device="cuda")] >> 32
            tgt = torch.randint(0, n, (nodes * OUT_EDGES,), generator=gen, device="cuda")
            out_e = torch.unique((new.repeat_interleave(OUT_EDGES) << 32) | tgt)
            in_e = torch.unique((src << 32) | new.repeat_interleave(IN_EDGES))
            link = torch.cat([_rows(out_e, 0), _rows(in_e, 0)])
            edit = torch.cat([edit, add, link[perm(link.shape[0])]])
            undo = torch.cat([undo, torch.stack([new, zero, torch.full_like(new, 3)], 1)])
        there, back = edit, undo
    return edges, seeds, there, back


class _Batch:
    """A batch as the engine takes it; new node ids follow the engine's count."""

    def __init__(self, rows, n, device):
        self.count = rows.shape[0]
        ops = rows.to(torch.int32)
        self.fresh = None
        if int((ops[:, :2] >= n).sum()):
            fresh = ops[:, :2] >= n
            self.fresh = (fresh, fresh.cpu().numpy())
        self.dev = ops.contiguous() if device else None
        self.host = None if device else ops.cpu().numpy().copy()
        self.base = n

    def apply(self, eng, eps, base):
        if self.fresh is not None and base != self.base:
            if self.dev is not None:
                self.dev[:, :2] += self.fresh[0] * (base - self.base)
                torch.cuda.current_stream().synchronize()
            else:
                self.host[:, :2] += self.fresh[1] * np.int32(base - self.base)
            self.base = base
        if self.dev is not None:
            eng.apply_updates_device(self.dev, self.count, eps)
        else:
            eng.apply_updates(self.host.view(N.UPDATE_DTYPE).reshape(-1), eps)


class _State:
    pass


def prepare(case, seed):
    """The engine with the graph loaded and the initial scores, and the batches."""
    st = _State()
    st.case = case
    edges, seeds, there, back = _draw_inputs(case, seed)
    u, v = (x.to(torch.int32).cpu().numpy() for x in _split(edges))
    st.stream = torch.cuda.Stream()
    one = case["seeds"] == 1
    st.eng = N.Engine(precision=PREC[case["prec"]], stream=st.stream.cuda_stream,
                      node_order=case["order"], use_graphs=case["graphs"],
                      deterministic=case["det"] and one,
                      max_nodes=case["n"] + (1_000_000 if case["nodes"] else 40_000))
    st.eng.load_graph(case["n"], u, v)
    st.eng.set_seeds(seeds.to(torch.int32).cpu().numpy(), C)
    if case["kind"] != "cpi":
        st.eng.init_scores(case["eps"] * 0.01)
    if case["kind"] == "update":
        st.there = _Batch(there, case["n"], case["device"])
        st.back = _Batch(back, case["n"], case["device"])
    if case["kind"] == "topk":
        st.m = min(32, case["seeds"])
        st.eng.query_slots(st.m)
    torch.cuda.synchronize()
    return st


def _read(st):
    """Every tracked score vector, as a program that hands them on takes them."""
    S, eng = st.case["seeds"], st.eng
    out = torch.empty(S, eng.num_nodes(), dtype=torch.float64, device="cuda")
    st.stream.synchronize()
    for j in range(S):
        eng.query_device(out[j], j)
    return out if st.case["prec"] == "f64" else out.float()


def run(st):
    case, eng = st.case, st.eng
    with torch.cuda.stream(st.stream):
        if case["kind"] == "topk":
            slots = range(st.m)
            eng.topk_async_many(slots, slots, case["k"])
            got = [eng.topk_wait(s) for s in slots]
            return {"ids": np.stack([i for i, _ in got]), "scores": np.stack([s for _, s in got])}
        if case["kind"] == "cpi":
            eng.init_scores(case["eps"])
            return {"scores": _read(st)}
        n, base, new = case["n"], eng.num_nodes(), case["nodes"]
        out = {}
        for name, batch in (("there", st.there), ("back", st.back)):
            batch.apply(eng, case["eps"], base)
            r = _read(st)
            out[name] = r[:, :n]
            if new and name == "there":  # this pass's nodes (those of earlier ones are gone)
                out["new"] = r[:, base:]
        return out


def work(case):
    """Each input read once, each output written once: per call the operations
    (12 bytes each), the in-lists (4 bytes an edge, 4 a node), the scores read
    and written (8 bytes each way) and every vector that is handed on; one sum
    over the in-lists per call is the least a change costs."""
    n, S = case["n"], case["seeds"]
    m = case["m"] * (2 if case["graph"] == "chunglu" else 1)
    out = 8 if case["prec"] == "f64" else 4
    if case["kind"] == "topk":
        j = min(32, S)
        return {"bytes": j * (8 * n + 12 * case["k"]), "flops": 0}
    if case["kind"] == "cpi":
        steps = max(1, int(math.log(case["eps"] / C) / math.log(1 - C)))
        return {"bytes": 4 * m + 4 * n + (8 + out) * n * S, "flops": 2 * m * S * steps}
    ops = case["ops"] * (2 if case["graph"] == "chunglu" else 1) + 17 * case["nodes"]
    return {"bytes": 2 * (12 * ops + 4 * m + 4 * n + (16 + out) * n * S), "flops": 4 * m * S}


# --------------------------------------------------------------------------
# The same in 64 bits, from the definition (Algorithm 1 of arXiv 1712.00595)
# --------------------------------------------------------------------------
def _matrix(keys, n):
    """(1-c) A~^T as a sparse matrix, A~ the row-normalised adjacency."""
    keys = torch.unique(keys)
    u, v = _split(keys)
    deg = torch.bincount(u, minlength=n)
    at = torch.argsort(v, stable=True)
    ptr = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    ptr[1:] = torch.cumsum(torch.bincount(v, minlength=n), 0)
    val = (1.0 - C) / deg[u[at]].double()
    return torch.sparse_csr_tensor(ptr, u[at], val, (n, n))


def _series(M, x, r, eps):
    """r + x(0) + x(1) + ..., each column until its first ||x(i)||_1 <= eps."""
    r += x
    live = x.abs().sum(0) > 0
    while bool(live.any()):
        x = M @ x
        r += x
        live &= x.abs().sum(0) > eps
        x *= live
    return r


def _edit(keys, rows, n):
    """The edge keys after a batch (insertions, deletions and node deletions)."""
    k = (rows[:, 0] << 32) | rows[:, 1]
    keys = torch.cat([keys[~torch.isin(keys, k[rows[:, 2] == 1])], k[rows[:, 2] == 0]])
    gone = torch.zeros(n, dtype=torch.bool, device="cuda")
    gone[rows[rows[:, 2] == 3, 0]] = True
    u, v = _split(keys)
    return torch.unique(keys[~gone[u] & ~gone[v]])


def exact(case, seed):
    edges, seeds, there, back = _draw_inputs(case, seed)
    n, S, new = case["n"], case["seeds"], case["nodes"]
    total = n + new
    eps = case["eps"]
    M = _matrix(edges, total)
    q = torch.zeros(total, S, dtype=torch.float64, device="cuda")
    q[seeds, torch.arange(S, device="cuda")] = C
    r = _series(M, q, torch.zeros_like(q), eps if case["kind"] == "cpi" else eps * 0.01)
    if case["kind"] == "cpi":
        return {"scores": r.T.contiguous()}
    if case["kind"] == "topk":
        best = torch.topk(r[:, : min(32, S)], case["k"], dim=0).values
        return {"ids": None, "scores": best.T.contiguous()}
    out, keys = {}, torch.unique(edges)
    for name, rows in (("there", there), ("back", back)):
        keys = _edit(keys, rows, total)
        M2 = _matrix(keys, total)
        r = _series(M2, M2 @ r - M @ r, r, eps)
        M = M2
        t = r.T.clone(memory_format=torch.contiguous_format)
        out[name] = t[:, :n]
        if new and name == "there":
            out["new"] = t[:, n:]
    return out
