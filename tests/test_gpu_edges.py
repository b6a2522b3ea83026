"""The one-seed kernel at the sizes where its step forms change hands, against
the oracle: in-lists around the stream, block and piece lengths, rows around
the push piece, frontiers of one node and of more nodes than warps, and pool
offsets in any order (lists rewritten by batches).

Tolerances are those of the parity tests (FP64 L1 1e-10; FP32 products 1e-5,
the oracle replaying the same step counts).
"""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1712_00595_gb300 import native as N
from paper_1712_00595_gb300 import workloads as W

pytestmark = pytest.mark.gpu

C_RESTART = 0.15
TOL = {N.OSP_PREC_FP64: 1e-10, N.OSP_PREC_FP32_ACC64: 1e-5}
LENGTHS = [0, 1, 2, 31, 32, 33, 63, 64, 65, 127, 128, 129, 255, 256, 257, 511, 513, 1023, 1024,
           1025, 1300, 2049]


def edge_graph(rng, n, chain):
    """Nodes 0.. have in-lists (chain = 0) or out-lists (1) of every length of
    LENGTHS, between others of 0..9 entries."""
    src, dst = [], []
    for v in range(n):
        k = LENGTHS[v // 3] if v % 3 == 0 and v // 3 < len(LENGTHS) else int(rng.integers(0, 10))
        u = rng.choice(n, min(k, n), replace=False)
        src += list(u) if not chain else [v] * u.size
        dst += [v] * u.size if not chain else list(u)
    return np.array(src, np.int32), np.array(dst, np.int32)


@pytest.mark.parametrize("prec", [N.OSP_PREC_FP64, N.OSP_PREC_FP32_ACC64])
@pytest.mark.parametrize("chain", [0, 1])
@pytest.mark.parametrize("n", [2300, 40011])
def test_list_lengths_at_the_edges_of_the_step_forms(prec, chain, n):
    rng = np.random.default_rng(n + chain)
    src, dst = edge_graph(rng, n, chain)
    seed = 3 * (len(LENGTHS) - 1)  # the longest row of the out-list graph
    eng = N.Engine(precision=prec, device=0)
    eng.load_graph(n, src, dst)
    eng.set_seeds([seed], C_RESTART)
    st = eng.init_scores(1e-13)
    g = O.Graph(n, src, dst)
    r, _, _ = O.cpi(*g.csr(), seed, C_RESTART, 1e-13, force_iters=st["iterations"])
    assert np.abs(eng.query() - r).sum() <= TOL[prec]
    # one op (a frontier of one row), then rewrites of many lists
    batches = W.edge_update_stream(src, dst, n, 1, 1, 0, seed=5)
    batches += W.edge_update_stream(np.concatenate([src, batches[0]["u"]]),
                                    np.concatenate([dst, batches[0]["v"]]), n, 2, 400, 400, seed=6)
    for ops in batches:
        st = eng.apply_updates(ops, 1e-12)
        old = g.csr()
        assert g.apply(ops) == -1
        r, _, _, _ = O.osp(old, g.csr(), r, C_RESTART, 1e-12, force_iters=st["iterations"])
        assert np.abs(eng.query() - r).sum() <= TOL[prec]
    eng.close()


def test_push_only_steps_reach_every_row_length():
    """push_alpha so small that every step pushes: frontiers from one node to
    all of them, rows of every length."""
    n = 9000
    rng = np.random.default_rng(8)
    src, dst = edge_graph(rng, n, 1)
    eng = N.Engine(precision=N.OSP_PREC_FP64, device=0, push_alpha=1e-9, push_beta=1e-9)
    eng.load_graph(n, src, dst)
    eng.set_seeds([3 * (len(LENGTHS) - 1)], C_RESTART)
    st = eng.init_scores(1e-12)
    assert st["push_iterations"] == st["iterations"]
    r, _, _ = O.cpi(*O.Graph(n, src, dst).csr(), 3 * (len(LENGTHS) - 1), C_RESTART, 1e-12,
                    force_iters=st["iterations"])
    assert np.abs(eng.query() - r).sum() <= 1e-10
    eng.close()


BF16, F32, F64 = N.OSP_PREC_BF16_ACC64, N.OSP_PREC_FP32_ACC64, N.OSP_PREC_FP64


@pytest.mark.parametrize("prec,S,group", [
    (BF16, 20, 0), (BF16, 64, 0), (BF16, 100, 32), (BF16, 100, 0), (BF16, 100, 128),
    (BF16, 200, 128), (BF16, 200, 256), (F32, 20, 0), (F32, 64, 0), (F32, 100, 0), (F32, 200, 64),
    (F32, 200, 256), (F64, 17, 0), (F64, 60, 32), (F64, 60, 0), (F64, 100, 128)])
def test_blocks_at_the_edges_of_the_row_stages(prec, S, group):
    """Seed blocks in every group width of the row rings (and past it, by lanes):
    in-lists around the 8- and 16-row stages, the 32-edge windows and the
    long-list pieces, in the oracle's lock-step, L1 <= 1e-10 (double) and 1e-5 a
    seed (the bounds of the seed-block tests)."""
    n = 2300
    rng = np.random.default_rng(S + group)
    src, dst = edge_graph(rng, n, 0)
    more = rng.integers(0, n, (2, 400))
    for k, v in ((7, 198), (8, 201), (15, 204), (16, 207), (17, 210), (47, 213), (48, 216), (49, 219)):
        u = rng.choice(n, k, replace=False)
        src, dst = np.append(src, u), np.append(dst, np.full(k, v))
    src, dst = np.append(src, more[0]).astype(np.int32), np.append(dst, more[1]).astype(np.int32)
    seeds = rng.permutation(n)[:S].astype(np.int32)
    eng = N.Engine(precision=prec, device=0, seed_group=group, node_order=S % 3 % 2)
    eng.load_graph(n, src, dst)
    eng.set_seeds(seeds, C_RESTART)
    eng.init_scores(1e-11)
    it0, _, _ = eng.get_seed_stats()
    tol = 1e-10 if prec == F64 else 1e-5
    g = O.Graph(n, src, dst)
    old = g.csr()
    pick = list(range(0, S, max(1, S // 12)))
    r = {j: O.cpi(*old, int(seeds[j]), C_RESTART, 1e-11, force_iters=int(it0[j]))[0] for j in pick}
    for ops in W.edge_update_stream(src, dst, n, 2, 300, 300, seed=S):
        eng.apply_updates(ops, 1e-9)
        assert g.apply(ops) == -1
        new = g.csr()
        it, _, _ = eng.get_seed_stats()
        for j in pick:
            r[j], _, _, _ = O.osp(old, new, r[j], C_RESTART, 1e-9, force_iters=int(it[j]))
            assert np.abs(eng.query(j) - r[j]).sum() <= tol
        old = new
    eng.close()


@pytest.mark.parametrize("n", [1, 255, 4097, 70001])
def test_topk_of_awkward_vectors(n):
    """Rankings where the radix passes, the collection and the one-CTA narrowing
    change hands: ties at the cut (ids decide), more equal keys than a sort
    holds, keys that differ in the last bits, k around 256 and at its limits."""
    torch = pytest.importorskip("torch")
    rng = np.random.default_rng(n)
    few = rng.integers(0, 3, n).astype(np.float64) * 0.25
    near = 1.0 + rng.integers(0, 7, n) * 2.0 ** -52
    wide = np.exp(rng.normal(-12, 6, n))
    zeros = np.zeros(n)
    zeros[rng.integers(0, n, min(n, 37))] = 0.5
    for v in (few, near, wide, zeros, np.full(n, 1.0 / n)):
        dv = torch.from_numpy(v).cuda()
        for k in (1, 100, 255, 256, 257, 1000, 4096):
            ids = torch.empty(k, dtype=torch.int32, device="cuda")
            sc = torch.empty(k, dtype=torch.float64, device="cuda")
            got = torch.zeros(1, dtype=torch.int32, device="cuda")
            N.topk_noalloc(dv, n, k, ids, sc, got, stream=torch.cuda.current_stream().cuda_stream)
            torch.cuda.synchronize()
            c = int(got)
            want_ids, want_sc = O.topk(v, k)
            assert c == min(n, k)
            assert np.array_equal(ids[:c].cpu().numpy(), want_ids)
            assert np.array_equal(sc[:c].cpu().numpy(), want_sc)


@pytest.mark.parametrize("n_ops", [511, 1024, 1025, 2500, 9000])
def test_batches_of_every_op_kind_across_the_ingest_sizes(n_ops):
    """Edge and node ops, row zeroings, repeated and contradicting ops, on both
    sides of the one-CTA ingest: the graph equals the oracle's, and an invalid op
    anywhere leaves it unchanged and is the one reported."""
    rng = np.random.default_rng(n_ops)
    n = 700
    src, dst = W.er_graph(n, 6000, 3)
    seed = 5
    eng = N.Engine(precision=N.OSP_PREC_FP64, device=0, max_nodes=n + 40000, use_graphs=n_ops % 2 == 0)
    eng.load_graph(n, src, dst)
    eng.set_seeds([seed], C_RESTART)
    eng.init_scores(1e-10)
    g = O.Graph(n, src, dst)
    nn, dead = n, set()
    for rep in range(3):
        kind = rng.choice(5, n_ops, p=[0.46, 0.46, 0.04, 0.02, 0.02])
        ops = np.zeros(n_ops, W.UPDATE_DTYPE)
        gone = set(dead)
        count = nn
        for i, k in enumerate(kind):
            live = [x for x in rng.integers(0, count, 40) if x not in gone]
            u, v = int(live[0]), int(live[1])
            if k <= 1 and rng.random() < 0.3:  # a few rows get many ops
                u = int(rng.integers(0, 12))
                u = u if u not in gone else int(live[0])
            if k == 3 and u == seed:
                k = 4
            ops[i] = (u, v, k) if k != 2 else (0, 0, 2)
            count += k == 2
            if k == 3:
                gone.add(u)
        bad = ops.copy()
        at = int(rng.integers(0, n_ops))
        bad[at] = [(count + 5, 0, 0), (0, -1, 1), (seed, 0, 3), (0, 0, 9)][rep % 4]
        before = eng.export_graph(0)
        st = eng.apply_updates(bad, 1e-8, allow=(N.OSP_EINVAL,))
        assert eng.last_status == N.OSP_EINVAL and st["bad_op"] == at
        assert all(np.array_equal(a, b) for a, b in zip(before, eng.export_graph(0)))
        eng.apply_updates(ops, 1e-8)
        assert g.apply(ops, protect=(seed,)) == -1
        nn, dead = count, gone
        ptr, idx = eng.export_graph(0)
        rp, col = g.csr()
        assert np.array_equal(ptr, rp) and np.array_equal(idx, col)
        ptr, idx = eng.export_graph(1)
        cp, row = g.csc()
        assert np.array_equal(ptr, cp) and np.array_equal(idx, row)
    eng.close()


@pytest.mark.parametrize("prec,S", [(F64, 20), (F64, 40), (F32, 100), (BF16, 200)])
def test_block_offsets_of_rows_that_grow_shrink_and_keep_their_length(prec, S):
    """Changed rows of every length around the offset piece: entries added,
    removed, exchanged one for one, and all taken out, in the oracle's lock-step,
    L1 <= 1e-10 (double) and 1e-5 a seed (the bounds of the seed-block tests)."""
    n = 2300
    rng = np.random.default_rng(S)
    src, dst = edge_graph(rng, n, 1)
    seeds = rng.permutation(n)[:S].astype(np.int32)
    eng = N.Engine(precision=prec, device=0)
    eng.load_graph(n, src, dst)
    eng.set_seeds(seeds, C_RESTART)
    eng.init_scores(1e-11)
    it0, _, _ = eng.get_seed_stats()
    g = O.Graph(n, src, dst)
    old = g.csr()
    pick = list(range(0, S, max(1, S // 10)))
    r = {j: O.cpi(*old, int(seeds[j]), C_RESTART, 1e-11, force_iters=int(it0[j]))[0] for j in pick}
    for turn in range(4):
        ptr, idx = (np.asarray(x) for x in old)
        ops = []
        for i in range(len(LENGTHS)):
            u = 3 * i
            has = idx[ptr[u]:ptr[u + 1]]
            lacks = np.setdiff1d(np.arange(n), has)
            k = {0: 3, 1: 1, 2: 40, 3: has.size}[(turn + i) % 4]
            if (turn + i) % 4 != 3:
                ops += [(u, int(v), 0) for v in rng.choice(lacks, min(k, lacks.size), replace=False)]
            if (turn + i) % 4 != 0:
                ops += [(u, int(v), 1) for v in rng.choice(has, min(k, has.size), replace=False)]
        ops = np.array(ops, W.UPDATE_DTYPE)
        eng.apply_updates(ops, 1e-9)
        assert g.apply(ops) == -1
        new = g.csr()
        it, _, _ = eng.get_seed_stats()
        for j in pick:
            r[j], _, _, _ = O.osp(old, new, r[j], C_RESTART, 1e-9, force_iters=int(it[j]))
            assert np.abs(eng.query(j) - r[j]).sum() <= (1e-10 if prec == F64 else 1e-5)
        old = new
    eng.close()


@pytest.mark.parametrize("det", [0, 1])
@pytest.mark.parametrize("n", [2, 607, 609, 4097, 622_591, 700_001])
def test_pull_plan_over_node_counts_around_its_ranges(n, det):
    """Every node in one task whatever the split of the nodes over the planning
    CTAs: few and many nodes a CTA, counts off the multiples of four, long lists
    first and last, against the oracle (L1 <= 1e-10)."""
    rng = np.random.default_rng(n)
    k = min(n, 3000)
    src = [rng.integers(0, n, 2 * n), rng.choice(n, k, replace=False), rng.choice(n, k, replace=False)]
    dst = [rng.integers(0, n, 2 * n), np.zeros(k, np.int64), np.full(k, n - 1)]
    e = np.unique(np.stack([np.concatenate(src), np.concatenate(dst)], 1), axis=0).astype(np.int32)
    src, dst = np.ascontiguousarray(e[:, 0]), np.ascontiguousarray(e[:, 1])
    eng = N.Engine(precision=N.OSP_PREC_FP64, device=0, deterministic=det)
    eng.load_graph(n, src, dst)
    eng.set_seeds([n // 2], C_RESTART)
    st = eng.init_scores(1e-9)
    g = O.Graph(n, src, dst)
    old = g.csr()
    r, _, _ = O.cpi(*old, n // 2, C_RESTART, 1e-9, force_iters=st["iterations"])
    assert np.abs(eng.query() - r).sum() <= 1e-10
    ops = np.array([(n - 1, 0, 1), (n // 2, n - 1, 0), (0, n // 3, 0)], W.UPDATE_DTYPE)
    st = eng.apply_updates(ops, 1e-9)
    assert g.apply(ops) == -1
    r, _, _, _ = O.osp(old, g.csr(), r, C_RESTART, 1e-9, force_iters=st["iterations"])
    assert np.abs(eng.query() - r).sum() <= 1e-10
    eng.close()


@pytest.mark.parametrize("n", [1, 2, 1023, 65536, 311_297])
@pytest.mark.parametrize("start", [0, 1])
def test_topk_of_a_vector_at_any_element(start, n):
    """Vectors that start at an even and at an odd element, whole and ragged passes
    of the paired loads, negative and infinite scores: exact."""
    torch = pytest.importorskip("torch")
    rng = np.random.default_rng(n + start)
    v = rng.normal(0, 1, n)
    v[rng.integers(0, n, 1 + n // 50)] = -0.0
    v[rng.integers(0, n)] = np.inf
    v[rng.integers(0, n)] = -np.inf
    buf = torch.zeros(n + 1, dtype=torch.float64, device="cuda")
    buf[start:start + n] = torch.from_numpy(v).cuda()
    for k in (1, 77, 3000):
        ids = torch.empty(k, dtype=torch.int32, device="cuda")
        sc = torch.empty(k, dtype=torch.float64, device="cuda")
        got = torch.zeros(1, dtype=torch.int32, device="cuda")
        N.topk_noalloc(buf[start:], n, k, ids, sc, got, stream=torch.cuda.current_stream().cuda_stream)
        torch.cuda.synchronize()
        c = int(got)
        assert c == min(n, k)
        key = np.where(np.signbit(v), ~v.view(np.uint64), v.view(np.uint64) | np.uint64(1 << 63))
        want = np.lexsort((np.arange(n), ~key))[:c]
        assert np.array_equal(ids[:c].cpu().numpy(), want)
        assert np.array_equal(sc[:c].cpu().numpy(), v[want])


@pytest.mark.parametrize("prec", [F64, F32])
def test_deterministic_norms_with_many_lists_in_pieces(prec):
    """Deterministic mode with 60 in-lists of two to nine pieces, whose |x| joins a
    step's norm apart from the CTAs' sums and is written again in the next step: the
    norm of every step agrees with the oracle's, and two contexts agree bit for bit.

    Relative bound of a step's norm, as in the parity tests: an entry rounds the stored
    value, the scale and the product once each, per-lane chains of at most 1,024 / 32
    terms, five warp levels and nine pieces (at most 50 u, u = 2^-24 or 2^-53); the
    oracle adds its in-edges in turn; the two norm sums add 2 n 2^-53."""
    rng = np.random.default_rng(17)
    n = 10_000
    src, dst = [rng.integers(0, n, 8 * n)], [rng.integers(0, n, 8 * n)]
    for v in range(60):
        src.append(rng.choice(n, int(rng.integers(1025, 9000)), replace=False))
        dst.append(np.full(src[-1].size, 3 * v))
    src, dst = np.concatenate(src).astype(np.int32), np.concatenate(dst).astype(np.int32)
    ops = W.edge_update_stream(src, dst, n, 1, 300, 300, seed=4)[0]
    runs = []
    for _ in range(2):
        eng = N.Engine(precision=prec, device=0, deterministic=True)
        eng.load_graph(n, src, dst)
        eng.set_seeds([1], C_RESTART)
        eng.init_scores(1e-11)
        runs.append([eng.get_l1_history(), eng.query()])
        eng.apply_updates(ops, 1e-11)
        runs[-1] += [eng.get_l1_history(), eng.query()]
        eng.close()
    for a, b in zip(*runs):
        assert a.shape == b.shape and np.array_equal(a.view(np.uint64), b.view(np.uint64))
    hist = runs[0][0]
    rp, col = O.Graph(n, src, dst).csr()
    want = O.cpi(rp, col, 1, C_RESTART, 1e-11, force_iters=hist.size - 1)[2]
    u = 2.0 ** -53 if prec == F64 else 2.0 ** -24
    d_in = int(np.bincount(col, minlength=n).max())
    delta = 50 * u + (d_in + 2) * 2.0 ** -53
    rtol = (1.0 + delta) ** np.arange(hist.size) - 1.0 + 2 * n * 2.0 ** -53
    assert np.all(np.abs(hist - want) <= rtol * want)


@pytest.mark.parametrize("S", [1, 3])
def test_large_batch_without_node_room_changes_nothing(S):
    """A batch of several sub-batches whose first one finds no node slots left is
    refused with OSP_ENOMEM: scores, graph and residual bound stay, bit for bit, the
    call's steps are those of a zero offset, and later batches go on from there."""
    n = 200
    src, dst = W.er_graph(n, 1500, 5)
    eng = N.Engine(precision=N.OSP_PREC_FP64, device=0, max_nodes=n)
    eng.load_graph(n, src, dst)
    eng.set_seeds(np.arange(S, dtype=np.int32), C_RESTART)
    eng.init_scores(1e-10)
    grow = np.zeros(300, W.UPDATE_DTYPE)  # room is left for a batch of 16,084 ops only
    grow["op"] = W.OP_ADD_NODE
    eng.apply_updates(grow, 1e-9)
    eng.apply_updates(W.edge_update_stream(src, dst, n, 1, 40, 40, seed=2)[0], 1e-9)
    rng = np.random.default_rng(4)
    big = np.zeros(20_000, W.UPDATE_DTYPE)
    big["u"], big["v"] = rng.integers(0, n, (2, big.size))
    before = [eng.query(j) for j in range(S)], eng.export_graph(0), eng.get_residual_bounds()
    for _ in range(20):
        st = eng.apply_updates(big, 1e-9, allow=(N.OSP_ENOMEM,))
        assert eng.last_status == N.OSP_ENOMEM
        assert st["iterations"] == 1 and st["qoff_l1"] == 0.0 and st["last_x_l1"] == 0.0
        assert np.array_equal(eng.get_l1_history(), [0.0, 0.0])
        assert np.array_equal(eng.get_residual_bounds(), before[2])
        for j in range(S):
            assert np.array_equal(eng.query(j), before[0][j])
        assert all(np.array_equal(a, b) for a, b in zip(eng.export_graph(0), before[1]))
    g = O.Graph(n, src, dst)
    g.apply(grow)
    g.apply(W.edge_update_stream(src, dst, n, 1, 40, 40, seed=2)[0])
    old = g.csr()
    ops = big[:3000]
    st = eng.apply_updates(ops, 1e-9)
    assert g.apply(ops) == -1
    it = eng.get_seed_stats()[0] if S > 1 else [st["iterations"]]
    for j in range(S):
        r = O.osp(old, g.csr(), before[0][j], C_RESTART, 1e-9, force_iters=int(it[j]))[0]
        assert np.abs(eng.query(j) - r).sum() <= 1e-10
    eng.close()


@pytest.mark.parametrize("fill", [0, 600])
@pytest.mark.parametrize("S", [1, 3])
def test_zeroed_rows_get_back_the_entries_at_the_edges_of_the_merge_pieces(S, fill):
    """A row zeroed and given back old entries in one batch, the entries around the
    256-entry pieces of the old list among them: in its own out-list (node 5) and as
    an entry of long in-lists (node 7's). Graph equal to the oracle's, scores L1 <=
    1e-10. fill: other ops, for the ingest over many CTAs."""
    rng = np.random.default_rng(fill)
    n = 1500
    src = [np.full(1100, 5), np.arange(8, 908), rng.integers(8, n, 6000)]
    dst = [np.arange(20, 1120), np.full(900, 7), rng.integers(8, n, 6000)]
    e = np.unique(np.stack([np.concatenate(src), np.concatenate(dst)], 1), axis=0).astype(np.int32)
    src, dst = np.ascontiguousarray(e[:, 0]), np.ascontiguousarray(e[:, 1])
    eng = N.Engine(precision=N.OSP_PREC_FP64, device=0)
    eng.load_graph(n, src, dst)
    eng.set_seeds(np.array([5, 0, 300][:S], np.int32), C_RESTART)
    eng.init_scores(1e-12)
    g = O.Graph(n, src, dst)
    old = g.csr()
    r = [O.cpi(*old, s, C_RESTART, 1e-12)[0] for s in [5, 0, 300][:S]]
    for turn in range(3):
        out5 = old[1][old[0][5]:old[0][6]]
        in7 = np.flatnonzero([7 in old[1][old[0][u]:old[0][u + 1]] for u in range(n)])
        back5 = out5[[i for i in (0, 254, 255, 256, 511, 512, 767, 1023) if i < out5.size]]
        ops = [(5, 0, 4)] + [(5, int(v), 0) for v in back5]
        for i in (254, 255, 256, 511, 512, 767):
            if i < in7.size and in7[i] != 5:
                ops += [(int(in7[i]), 0, 4), (int(in7[i]), 7, 0)]
        # node 5 gets a long row again for the next turn
        more = [(5, int(v), 0) for v in rng.choice(np.arange(20, n), 700, replace=False)]
        more += [(int(u), int(v), 0) for u, v in rng.integers(8, n, (fill, 2))]
        for batch in (ops, more) if turn % 2 else (ops + more[700:], more):
            batch = np.array(batch, W.UPDATE_DTYPE)
            st = eng.apply_updates(batch, 1e-12)
            assert g.apply(batch) == -1
            new = g.csr()
            assert all(np.array_equal(a, b) for a, b in zip(eng.export_graph(0), new))
            assert all(np.array_equal(a, b) for a, b in zip(eng.export_graph(1), g.csc()))
            it = eng.get_seed_stats()[0] if S > 1 else [st["iterations"]]
            for j in range(S):
                r[j] = O.osp(old, new, r[j], C_RESTART, 1e-12, force_iters=int(it[j]))[0]
                assert np.abs(eng.query(j) - r[j]).sum() <= 1e-10
            old = new
    eng.close()


@pytest.mark.parametrize("prec,S,kw", [
    (F64, 17, {}), (F64, 100, dict(seed_group=128)), (F32, 100, {}), (F32, 40, dict(seed_gather=1)),
    (F32, 40, dict(seed_gather=2)), (BF16, 100, {}), (BF16, 40, dict(seed_gather=2))])
def test_block_norms_of_a_call_are_the_largest_of_its_seeds(prec, S, kw):
    """qoff_l1, last_x_l1 and the step history of a seed block are the maxima of the
    per-seed norms (all below 1), to the bit."""
    n = 1500
    src, dst = W.er_graph(n, 12_000, 6)
    eng = N.Engine(precision=prec, device=0, **kw)
    eng.load_graph(n, src, dst)
    eng.set_seeds(np.random.default_rng(1).permutation(n)[:S].astype(np.int32), C_RESTART)
    sts = [eng.init_scores(1e-6)]
    for ops in [None] + W.edge_update_stream(src, dst, n, 2, 60, 60, seed=3):
        if ops is not None:
            sts.append(eng.apply_updates(ops, 1e-6))
        it, q, last = eng.get_seed_stats()
        hist = eng.get_l1_history()
        assert hist.size == sts[-1]["iterations"] + 1 and np.all(hist > 0) and np.all(hist < 1)
        assert hist[0] == sts[-1]["qoff_l1"] == q.max()
        assert hist[-1] == sts[-1]["last_x_l1"] == last[it == it.max()].max()
    eng.close()


@pytest.mark.parametrize("S,group,gather", [(20, 0, 0), (64, 0, 0), (100, 0, 0), (200, 256, 0), (40, 0, 2)])
def test_norms_of_float_blocks_are_sums_in_double(S, group, gather):
    """FP32 seed blocks: ||x(k)||_1 against the double sum of |x(k)|, taken as the
    difference of the scores after k and after k - 1 steps (no list is long enough to
    be cut, so both runs add the same floats). Bound: the scores round at most
    2^-53 ||r||_1 = 2^-53 a step, 2 k of them; the sums of n terms 2 n 2^-53 relative."""
    n, k = 3000, 4
    src, dst = W.er_graph(n, 30_000, 9)
    eng = N.Engine(precision=F32, device=0, seed_group=group, seed_gather=gather)
    eng.load_graph(n, src, dst)
    eng.set_seeds(np.random.default_rng(S).permutation(n)[:S].astype(np.int32), C_RESTART)
    r = []
    for steps in (k - 1, k):
        eng.set_fixed_iterations(steps)
        eng.init_scores(1e-9)
        r.append([eng.query(j) for j in range(S)])
    _, _, last = eng.get_seed_stats()
    for j in range(S):
        want = np.abs(r[1][j] - r[0][j]).sum()
        assert abs(last[j] - want) <= 2 * k * 2.0 ** -53 + 2 * n * 2.0 ** -53 * want
    eng.close()


@pytest.mark.parametrize("S,kw", [(5, {}), (64, {}), (100, {}), (5, dict(seed_gather=2))])
def test_float_blocks_keep_subnormal_steps(S, kw):
    """A chain of 13 nodes, each with 2,000 out-edges: x falls by 0.85 / 2000 a step,
    past the smallest normal float (2^-126) at the twelfth. Every score is the oracle's
    within a step's float rounding: 13 x 4 roundings of 2^-24 relative, and 13 x 2 of
    the subnormal grid's half unit, 2^-150."""
    levels, fan = 13, 2000
    n = levels + fan
    src, dst = [], []
    for i in range(levels - 1):
        src += [i] * fan
        dst += [i + 1] + list(range(levels, n - 1))
    src, dst = np.array(src, np.int32), np.array(dst, np.int32)
    seeds = np.concatenate([[0], levels + np.arange(S - 1)]).astype(np.int32)
    eng = N.Engine(precision=F32, device=0, **kw)
    eng.load_graph(n, src, dst)
    eng.set_seeds(seeds, C_RESTART)
    eng.set_fixed_iterations(levels)
    eng.init_scores(1e-9)
    want = O.cpi(*O.Graph(n, src, dst).csr(), 0, C_RESTART, 1e-9, force_iters=levels)[0]
    assert 0 < want[levels - 1] < 2.0 ** -126
    got = eng.query(0)
    assert np.all(np.abs(got - want) <= 4 * levels * 2.0 ** -24 * want + levels * 2.0 ** -149)
    eng.close()


@pytest.mark.parametrize("prec,S,group", [
    (F64, 20, 0), (F64, 60, 0), (F32, 20, 0), (F32, 40, 64), (F32, 100, 0), (BF16, 20, 0), (BF16, 64, 0),
    (BF16, 200, 128)])
def test_register_gathers_are_taken_where_asked_for(prec, S, group):
    """seed_gather 1 in the group widths that the row rings serve by default: its own
    schedule is in force, and the scores follow the oracle's lock-step, L1 <= 1e-10
    (double) and 1e-5 a seed (the bounds of the seed-block tests)."""
    n = 2300
    rng = np.random.default_rng(S)
    src, dst = edge_graph(rng, n, 0)
    seeds = rng.permutation(n)[:S].astype(np.int32)
    eng = N.Engine(precision=prec, device=0, seed_gather=N.SEED_GATHER_REGISTERS, seed_group=group)
    eng.load_graph(n, src, dst)
    eng.set_seeds(seeds, C_RESTART)
    assert eng.get_schedule() == (1024, 256, 256, 4)
    eng.init_scores(1e-11)
    it, _, _ = eng.get_seed_stats()
    tol = 1e-10 if prec == F64 else 1e-5
    g = O.Graph(n, src, dst)
    old = g.csr()
    pick = list(range(0, S, max(1, S // 8)))
    r = {j: O.cpi(*old, int(seeds[j]), C_RESTART, 1e-11, force_iters=int(it[j]))[0] for j in pick}
    for ops in W.edge_update_stream(src, dst, n, 2, 300, 300, seed=S):
        eng.apply_updates(ops, 1e-9)
        assert g.apply(ops) == -1
        it, _, _ = eng.get_seed_stats()
        for j in pick:
            r[j], _, _, _ = O.osp(old, g.csr(), r[j], C_RESTART, 1e-9, force_iters=int(it[j]))
            assert np.abs(eng.query(j) - r[j]).sum() <= tol
        old = g.csr()
    eng.close()


@pytest.mark.parametrize("graphs", [0, 1])
@pytest.mark.parametrize("n_ops", [512, 513, 16383, 16384])
def test_batches_at_the_limits_of_the_ingest_routes(n_ops, graphs):
    """The last batch size of the one-CTA ingest and the first of the one over many
    CTAs, and the largest batches, whose last op (a node op at position 16,383) has the
    highest key of all: graph equal to the oracle's; each kind of invalid op, an unknown
    code among them, at the first, a middle and the last position is the one reported
    and leaves the graph as it was."""
    rng = np.random.default_rng(n_ops)
    n = 900
    src, dst = W.er_graph(n, 8000, 3)
    seed = 5
    eng = N.Engine(precision=F64, device=0, max_nodes=n + 60_000, use_graphs=graphs)
    eng.load_graph(n, src, dst)
    eng.set_seeds([seed], C_RESTART)
    eng.init_scores(1e-8)
    g = O.Graph(n, src, dst)
    nn = n
    for last in (2, 3, 4):
        ops = np.zeros(n_ops, W.UPDATE_DTYPE)
        ops["op"] = rng.choice([0, 1, 2, 4], n_ops, p=[0.49, 0.49, 0.01, 0.01])
        count = nn + np.cumsum(ops["op"] == 2) - (ops["op"] == 2)  # nodes before each op
        ops["u"] = 10 + (rng.random(n_ops) * (count - 10)).astype(np.int32)
        ops["v"] = 10 + (rng.random(n_ops) * (count - 10)).astype(np.int32)
        few = rng.random(n_ops) < 0.2  # a few rows get many ops
        ops["u"][few] = rng.integers(10, 20, few.sum())
        ops[-1] = (6 + last % 2, 0, last)  # ids below 10 take no other op
        before = eng.export_graph(0)
        for k, (at, op) in enumerate([(0, (nn + 70_000, 0, 0)), (n_ops // 2, (0, -1, 1)),
                                      (n_ops - 1, (seed, 0, 3)), (n_ops - 1, (0, 0, 9)),
                                      (n_ops // 3, (0, 0, -1))]):
            bad = ops.copy()
            bad[at] = op
            st = eng.apply_updates(bad, 1e-6, allow=(N.OSP_EINVAL,))
            assert eng.last_status == N.OSP_EINVAL and st["bad_op"] == at, (k, at)
        assert all(np.array_equal(a, b) for a, b in zip(before, eng.export_graph(0)))
        eng.apply_updates(ops, 1e-6)
        assert g.apply(ops, protect=(seed,)) == -1
        nn += int((ops["op"] == 2).sum())
        assert all(np.array_equal(a, b) for a, b in zip(eng.export_graph(0), g.csr()))
        assert all(np.array_equal(a, b) for a, b in zip(eng.export_graph(1), g.csc()))
        # node 7 was deleted in the second turn, node 6 is emptied in the third
    eng.close()


def sum_graph(rng, S, lengths, reps, row, max_degree, n):
    """S seeds with `row` out-edges each into a pool of nodes, lists of the given lengths
    drawn from the pool, pool nodes with out-degrees up to max_degree (spread over their
    logarithm). Returns the edges and {length: nodes}."""
    pool0 = S + reps * len(lengths)
    pool = np.arange(pool0, n)
    src = [np.repeat(np.arange(S), row)]
    dst = [np.concatenate([rng.choice(pool, row, replace=False) for _ in range(S)])]
    lists, v = {}, S
    for k in lengths:
        for _ in range(reps):
            src.append(rng.choice(pool, k, replace=False))
            dst.append(np.full(k, v))
            lists.setdefault(k, []).append(v)
            v += 1
    deg = np.exp(rng.uniform(0, np.log(max_degree), pool.size)).astype(int)
    src.append(np.repeat(pool, deg))
    dst.append(rng.choice(pool, deg.sum()))
    e = np.unique(np.stack([np.concatenate(src), np.concatenate(dst)], 1), axis=0).astype(np.int32)
    return np.ascontiguousarray(e[:, 0]), np.ascontiguousarray(e[:, 1]), lists


def row_sum_errors(got, y, src, dst, nodes):
    """(got - sum of the in-list's y) / sum |y|, signed so that a sum too small in size is
    negative, for every seed and node; the sums exact enough at twice the precision."""
    out = []
    for v in nodes:
        part = y[:, src[dst == v]].astype(np.longdouble)
        s, m = part.sum(1), np.abs(part).sum(1)
        ok = m > 0
        out.append(((got[ok, v] - s[ok]) / m[ok] * np.sign(s[ok])).astype(np.float64))
    return np.concatenate(out)


@pytest.mark.parametrize("S", [20, 40])
def test_double_row_sums_are_not_one_chain(S):
    """Lists of equal values 2^-12 fl(0.75 / 7), whose additions to a long sum all round the
    same way: one chain of 500 is off by 86 units of 2^-53. Sums by stages of at most 16
    rows, 16 stages a part, four parts, two pieces: at most 16 + 16 + 4 + 3 additions deep,
    half a unit in the last place (2^-53 relative) each."""
    from fractions import Fraction
    n, row = 1800, 768
    src, dst = [np.repeat(np.arange(S), row)], [np.tile(np.arange(900, 900 + row), S)]
    lists = (300, 500, 512, 767)
    for i, k in enumerate(lists):
        src.append(np.arange(900, 900 + k))
        dst.append(np.full(k, 100 + i))
    for u in range(900, 900 + row):  # every pool node: seven out-edges
        have = sum(u < 900 + k for k in lists)
        src.append(np.full(7 - have, u))
        dst.append(200 + (u + np.arange(7 - have)) % 300)
    src, dst = np.concatenate(src).astype(np.int32), np.concatenate(dst).astype(np.int32)
    eng = N.Engine(precision=F64, device=0)
    eng.load_graph(n, src, dst)
    eng.set_seeds(np.arange(S, dtype=np.int32), 0.25)
    eng.set_fixed_iterations(2)
    eng.init_scores(1e-9)
    y = Fraction(0.75 / 7) / 2 ** 12  # 0.25 x (0.75 / 768), exact, times fl(0.75 / 7)
    for j in (0, S - 1):
        r = eng.query(j)
        for i, k in enumerate(lists):
            assert abs(Fraction(float(r[100 + i])) / (k * y) - 1) <= Fraction(39, 2 ** 53), (j, k)
    eng.close()


@pytest.mark.parametrize("prec,S", [(F32, 40), (F32, 100), (BF16, 100)])
def test_float_row_sums_of_long_lists(prec, S):
    """Second step from scratch (float rows, also of a bf16 block): lists of 1,000 and 1,024
    rows against the double sum. An addition to a partial sum s rounds by at most 2^-24 s,
    as a random variable with a deviation of 2^-24 s / sqrt(3). Sums by stages of 8 or 16
    rows, 16 stages a part: the parts' sums, (2/8)^2 + .. + (8/8)^2 = 3.2, the stages within
    the parts 0.7 more, rows within stages and pieces less than 0.6: a deviation of
    sqrt(4.5 / 3) = 1.2 units of 2^-24, a mean size of 0.8 times that, 1.0. (A chain of 125
    stage sums: 3.0.) Rows of at most 64 columns take one chain of 32 stages of 16 rows in
    each piece of 512: 2 (1/2)^2 (11.3) = 5.7 and 1.3 for the rest, of which half is left when
    s counts with its place between two powers of two: sqrt(3.5 / 3) times 0.8, 0.9."""
    rng = np.random.default_rng(S)
    n = 6000
    src, dst, lists = sum_graph(rng, S, (1000, 1024), 8, 3000, 400, n)
    eng = N.Engine(precision=prec, device=0)
    eng.load_graph(n, src, dst)
    eng.set_seeds(np.arange(S, dtype=np.int32), C_RESTART)
    eng.set_fixed_iterations(2)
    eng.init_scores(1e-9)
    got = np.stack([eng.query(j) for j in range(S)])
    eng.close()
    d = np.bincount(src, minlength=n)
    scale = np.where(d > 0, (1 - C_RESTART) / np.maximum(d, 1), 0.0).astype(np.float32)
    x = np.zeros((S, n), np.float32)
    for j in range(S):
        x[j, dst[src == j]] = np.float32(C_RESTART) * scale[j]
    for k, nodes in lists.items():
        err = row_sum_errors(got, x * scale, src, dst, nodes) * 2.0 ** 24
        assert np.abs(err).mean() <= 1.0, (k, np.abs(err).mean())


@pytest.mark.parametrize("S", [20, 40, 100])
def test_bf16_row_sums_of_long_lists_are_not_truncated(S):
    """First step of a batch, bf16 rows over many decades: sums of 500 to 1,024 rows against
    the double sum of the stored rows. Sums that round to nearest have a mean error of zero;
    half a unit of 2^-24 is allowed. (Chains of up to 64 tensor-core additions, which drop
    what does not fit, came out 1.5 to 2.2 units small.)"""
    rng = np.random.default_rng(S)
    n = 5000
    src, dst, lists = sum_graph(rng, S, (500, 1000, 1024), 12, 2500, 1000, n)
    eng = N.Engine(precision=BF16, device=0)
    eng.load_graph(n, src, dst)
    eng.set_seeds(np.arange(S, dtype=np.int32), C_RESTART)
    eng.init_scores(1e-10)
    r0 = np.stack([eng.query(j) for j in range(S)])
    rows = np.concatenate([np.arange(S), rng.choice(np.arange(n // 2, n), 600, replace=False)])
    out = {u: dst[src == u] for u in rows.tolist()}
    ops = np.zeros(rows.size, W.UPDATE_DTYPE)  # one new edge a row, into the upper half
    for i, (u, t) in enumerate(out.items()):
        ops[i] = (u, rng.choice(np.setdiff1d(np.arange(n // 2, n), t)), 0)
    eng.set_fixed_iterations(1)
    eng.apply_updates(ops, 1e-9)
    got = np.stack([eng.query(j) for j in range(S)])
    eng.close()
    x = np.zeros((S, n))
    for op, (u, t) in zip(ops, out.items()):
        x[:, t] += (0.85 / (t.size + 1) - 0.85 / t.size) * r0[:, u:u + 1]
        x[:, op["v"]] += 0.85 / (t.size + 1) * r0[:, u]
    src, dst = np.concatenate([src, ops["u"]]), np.concatenate([dst, ops["v"]])
    d = np.bincount(src, minlength=n)
    scale = np.where(d > 0, 0.85 / np.maximum(d, 1), 0.0).astype(np.float32)
    b = (x.astype(np.float32) * scale).view(np.uint32).astype(np.uint64)
    y = (((b + 0x7FFF + ((b >> 16) & 1)) >> 16) << 16).astype(np.uint32).view(np.float32)  # to bf16
    for k, nodes in lists.items():
        err = row_sum_errors(got - r0 - x, y, src, dst, nodes) * 2.0 ** 24
        assert abs(err.mean()) <= 0.5, (k, err.mean())


@pytest.mark.parametrize("order", [0, 1])
@pytest.mark.parametrize("n", [2, 40_001, 900_001])
def test_columns_of_a_block_in_either_form_of_the_query(n, order):
    """A seed block's columns, small ones and those whose lines exceed the L2: the query of
    each column equals the rankings' scores (gathered by another kernel), to the bit, and
    the device query the host query."""
    torch = pytest.importorskip("torch")
    rng = np.random.default_rng(n)
    S = min(n, 5)
    src, dst = rng.integers(0, n, (2, 2 * n)).astype(np.int32)
    eng = N.Engine(precision=F32, device=0, node_order=order)
    eng.load_graph(n, src, dst)
    eng.set_seeds(rng.choice(n, S, replace=False).astype(np.int32), C_RESTART)
    eng.init_scores(1e-4)
    eng.query_slots(S)
    eng.topk_async_many(range(S), range(S), 500)
    out = torch.empty(n, dtype=torch.float64, device="cuda")
    for j in range(S):
        ids, sc = eng.topk_wait(j)
        r = eng.query(j)
        want_ids, want_sc = O.topk(r, 500)
        assert np.array_equal(ids, want_ids) and np.array_equal(sc, want_sc)
        eng.query_device(out, j)
        assert np.array_equal(out.cpu().numpy(), r)
    eng.close()
