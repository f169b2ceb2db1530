"""Every pair of accesses to shared memory that depend on each other has a wait between them, whatever the speed of the warps.  Kernels
run on a CPU thread by thread with vector clocks (cta.h), their results against the oracle's: the Phase-1 kernel of few problems at one
and two warps, one and two ranks a lane, ends on every iteration of a group of eight, iterations looked at one by one, folds and
hand-backs; the one of batches of up to 32 ranks; the one on classes of ranks where several lanes hold copies of a class; the rounds of the auction in one warp; the reassignment of chunks with no split, with splits located one by one and with splits located together."""
import ctypes

import numpy as np
import pytest

import cta
import oracle as O


@pytest.fixture(scope="module")
def so(tmp_path_factory):
    return cta.load(str(tmp_path_factory.mktemp("cta")), "cta_split.cpp", ["sinkhorn_split.cuh", "sinkhorn_common.cuh", "taot_internal.cuh"])


def test_a_vote_orders_no_memory_and_a_barrier_does(so):
    so.cta_reset()
    so.cta_exchange(1)
    assert so.cta_races() == 0 and so.cta_stuck() == 0
    so.cta_exchange(0)
    assert so.cta_races() > 0
    so.cta_reset()


def _loads(g, R, hot, cold):
    s, d = np.zeros((1, R), np.float32), np.zeros((1, R), np.float32)
    s[0, g.permutation(R)[:hot]] = g.integers(1, 4000, hot)
    free = np.flatnonzero(s[0] == 0) if hot + cold <= R else np.arange(R)
    d[0, free[:cold]] = g.integers(1, 900, cold)
    d *= s.sum() / d.sum()
    return s, d


def _solve(run, R, s, d, C, eps):
    """run(*pointers of s, d, C, the rows' log-sum-exp, 1 / eps, plan, iterations, row error, status) -> plan, iterations"""
    B = len(s)
    x = -C.astype(np.float64) / eps
    lse0 = np.log(np.exp(x - x.max(1, keepdims=True)).sum(1)) + x.max(1)
    plan = np.full((B, R, R), np.nan, np.float32)
    its, err, info = np.full(B, -9, np.int32), np.zeros(B, np.float32), np.zeros(B, np.int32)
    at = lambda a: a.ctypes.data_as(ctypes.c_void_p)
    run((at(s), at(d), at(C), at(lse0), ctypes.c_double(1.0 / np.float64(np.float32(eps)))), (at(plan), at(its), at(err), at(info)))
    return plan, its


def _check_plan(plan, s, d, C, eps, its):
    want = O.sinkhorn(s, d, C, eps, int(its), 0.0, 1, 1e-8)["plan"]
    assert (np.abs(plan - want) <= 1e-4 * np.maximum(want, 1e-7 * s.sum() / s.size ** 2)).all()


@pytest.mark.parametrize("R,hot,cold,threads", [(8, 3, 5, 128), (24, 9, 15, 128), (32, 20, 32, 128), (48, 16, 32, 128), (48, 16, 32, 64),
                                                (40, 18, 40, 128), (64, 20, 44, 128), (64, 31, 33, 128), (64, 20, 44, 64), (64, 40, 24, 128)])
@pytest.mark.parametrize("iters,tol,check_every", [(25, 0.0, 1), (120, 1e-3, 1), (120, 1e-3, 3), (30, 1e-9, 1),
                                                   (200, 3.5e-8, 8)])       # near what fp32 sums leave: met, and missed where it is asked
@pytest.mark.parametrize("eps", [0.05, 2.0])             # 0.05: folds
def test_few_problems(so, R, hot, cold, threads, iters, tol, check_every, eps):
    g = np.random.default_rng(R + hot + iters)
    C = (1.0 + 7.0 * g.random((R, R))).astype(np.float32)
    np.fill_diagonal(C, 0.0)
    s, d = _loads(g, R, hot, cold)
    so.cta_reset()
    plan, its = _solve(lambda i, o: so.cta_sinkhorn(1, R, threads, *i, iters, ctypes.c_float(tol), check_every, *o), R, s, d, C, eps)
    assert so.cta_races() == 0, so.cta_first().decode()
    assert so.cta_stuck() == 0
    if hot > 32:
        assert its[0] == -1
    elif its[0] == -1:                                   # handed back: a sum out of fp32's comfortable range
        assert eps == 0.05
    else:
        _check_plan(plan[0], s[0], d[0], C, eps, its[0])


@pytest.fixture(scope="module")
def tile(tmp_path_factory):
    return cta.load(str(tmp_path_factory.mktemp("cta")), "cta_tile.cpp", ["sinkhorn_tile.cuh", "sinkhorn_common.cuh", "taot_internal.cuh"])


@pytest.mark.parametrize("R,hot,cold", [(8, 3, 5), (24, 9, 15), (32, 20, 12), (32, 15, 17)])
@pytest.mark.parametrize("iters,tol,check_every", [(40, 0.0, 1), (120, 1e-3, 1), (120, 1e-3, 3)])
@pytest.mark.parametrize("eps", [0.05, 2.0])             # 0.05: folds
def test_batches_of_problems(tile, R, hot, cold, iters, tol, check_every, eps):
    g = np.random.default_rng(R + hot + iters)
    C = (1.0 + 7.0 * g.random((R, R))).astype(np.float32)
    np.fill_diagonal(C, 0.0)
    s, d = _loads(g, R, hot, cold)
    tile.cta_reset()
    plan, its = _solve(lambda i, o: tile.cta_sinkhorn(1, R, *i, iters, ctypes.c_float(tol), check_every, *o), R, s, d, C, eps)
    assert tile.cta_races() == 0, tile.cta_first().decode()
    assert tile.cta_stuck() == 0
    if its[0] == -1:
        assert eps == 0.05
    else:
        _check_plan(plan[0], s[0], d[0], C, eps, its[0])


@pytest.fixture(scope="module")
def classes(tmp_path_factory):
    return cta.load(str(tmp_path_factory.mktemp("cta")), "cta_class.cpp", ["sinkhorn_class.cu", "sinkhorn_class.h", "sinkhorn_common.cuh", "taot_internal.cuh"])


@pytest.mark.parametrize("R,node,nc", [(64, 8, 8), (64, 32, 2)])
@pytest.mark.parametrize("B,share", [(1, 0), (5, 1)])
@pytest.mark.parametrize("iters,tol", [(60, 0.0), (200, 1e-6)])
@pytest.mark.parametrize("eps", [0.05, 2.0])             # 0.05: folds
def test_classes_of_ranks(classes, R, node, nc, B, share, iters, tol, eps):
    g = np.random.default_rng(R + node + B)
    at = np.arange(R) // node
    C = np.where(at[:, None] == at[None, :], 1.0, np.where(at[:, None] // 4 == at[None, :] // 4, 6.0, 16.0)).astype(np.float32)
    np.fill_diagonal(C, 0.0)
    loads = [_loads(g, R, 10 + b, 40 - b) for b in range(B)]
    s, d = (np.concatenate(x) for x in zip(*loads))
    classes.cta_reset()

    def run(i, o):
        assert classes.cta_classes(B, R, share, *i, iters, ctypes.c_float(tol), *o) == nc
    plan, its = _solve(run, R, s, d, C, eps)
    assert classes.cta_races() == 0, classes.cta_first().decode()
    assert classes.cta_stuck() == 0
    for b in range(B):
        assert its[b] > 0
        _check_plan(plan[b], s[b], d[b], C, eps, its[b])


@pytest.fixture(scope="module")
def assign(tmp_path_factory):
    return cta.load(str(tmp_path_factory.mktemp("cta")), "cta_assign.cpp", ["assign.cu", "taot_internal.cuh"])


@pytest.mark.parametrize("fed", [0, 1, 2, 4, 5, 14])     # slots a rank feeds; up to four splits of a chunk are located one by one
@pytest.mark.parametrize("seg,vec", [(900, 1), (1037, 0)])
@pytest.mark.parametrize("threads", [256, 512])
def test_reassignment_of_a_chunk(assign, fed, seg, vec, threads):
    R, E, K, chunk = 2, 5, 8, 16384
    S, nc = R * K, -(-seg // chunk)
    g = np.random.default_rng(fed + seg)
    topk = g.integers(0, E, (1, R, seg)).astype(np.int32)
    cc = np.zeros((1, R, nc, E), np.int32)
    X = np.zeros((1, R, S), np.int32)
    slots = g.integers(0, E, S).astype(np.int32)
    for r in range(R):
        for c in range(nc):
            cc[0, r, c] = np.bincount(topk[0, r, c * chunk:(c + 1) * chunk], minlength=E)
        X[0, r, g.permutation(S)[:fed]] = g.integers(1, seg // (E * 6), fed)
    out, info = np.full_like(topk, -7), np.zeros(1, np.int32)
    at = lambda a: a.ctypes.data_as(ctypes.c_void_p)
    assign.cta_reset()
    assign.cta_assign(1, R, E, K, ctypes.c_long(R * seg), ctypes.c_long(seg), nc, vec, threads, at(topk), at(cc), at(slots), at(X), at(out), at(info))
    assert assign.cta_races() == 0, assign.cta_first().decode()
    assert assign.cta_stuck() == 0
    assert (out.ravel() == O.assign(topk.reshape(R * seg, 1), R, E, K, slots, X[0]).ravel()).all()


@pytest.fixture(scope="module")
def auction(tmp_path_factory):
    return cta.load(str(tmp_path_factory.mktemp("cta")), "cta_auction.cpp", ["auction.cuh", "taot_internal.cuh"])


@pytest.mark.parametrize("R,D", [(32, 6), (64, 4)])      # one word of ranks and two; at most 32 classes
@pytest.mark.parametrize("lean,far,step", [(1, 12.0, 0.1), (0, 12.0, 0.1), (0, 2.0, 0.125)])     # the last: equal scores
@pytest.mark.parametrize("seed", [0, 1])
def test_auction_in_one_warp(auction, R, D, lean, far, step, seed):
    K, W, node = 2, R // 32, 8
    S = R * K
    g = np.random.default_rng(seed)
    at = np.arange(R) // node
    C = np.where(at[:, None] == at[None, :], 1.0, far).astype(np.float32)
    np.fill_diagonal(C, 0.0)
    B = O.default_preference(C)
    B3 = np.where(np.eye(R, dtype=bool), np.float32(1), B)                       # [rank, host]
    n = (g.integers(0, 60, (R, D)) * (g.random((R, D)) < 0.7)).astype(np.int32)
    slot_e = np.concatenate([g.permutation(D)[:K] for _ in range(R)]).astype(np.int32)
    tokens = (g.integers(1, 200, S) * (g.random(S) < 0.7)).astype(np.int32)
    # the (tier, win count) pairs, best score first
    tiers = np.unique(B3)[::-1].astype(np.float32)
    pairs = sorted(((t, w) for t in range(len(tiers)) for w in range(S + 1)),
                   key=lambda p: -(tiers[p[0]] - np.float32(step) * np.float32(p[1])))
    score = [tiers[t] - np.float32(step) * np.float32(w) for t, w in pairs]
    lst, ent = np.zeros(len(pairs), np.uint32), np.zeros((len(tiers), S + 1), np.uint32)
    for i, (t, w) in enumerate(pairs):
        tie = i + 1 < len(pairs) and score[i + 1] == score[i]
        above = len({float(tiers[q] - np.float32(step) * np.float32(w)) for q in range(t)} - {float(score[i])})
        lst[i] = w << 8 | t | (tie << 31)
        ent[t, w] = i << 16 | tie << 14 | above << 11 | w
    assert lean == 0 or not (lst >> 31).any()
    # classes: live slots of an expert on hosts of a node
    lead, nxt, of = [], np.full(S + 1, S, np.uint16), {}
    for s in range(S):
        if tokens[s]:
            key = (slot_e[s], at[s // K])
            if key in of:
                nxt[of[key]] = s
            else:
                lead.append(s)
            of[key] = s
    assert 16 < len(lead) <= 32
    a = np.append(tokens, 0).astype(np.int32)
    rec = np.stack([nxt.astype(np.uint32), a[nxt].astype(np.uint32)], 1)
    bits = lambda m: np.packbits(m.reshape(W, 32), axis=1, bitorder="little").view(np.uint32).ravel()
    avail = np.stack([bits(n[:, e] > 0) for e in range(D)], 1).astype(np.uint32)             # [W][D]
    lvl = np.zeros((W, S + 1), np.uint32)
    lvl[:, 0] = 0xFFFFFFFF
    tm, tw = np.zeros((len(tiers), W, S), np.uint32), np.zeros((len(tiers), S, 2), np.uint32)
    for t, value in enumerate(tiers):
        for c, s in enumerate(lead):
            tm[t, :, c] = bits(B3[:, s // K] == value)
            words = np.flatnonzero(tm[t, :, c])
            tw[t, c] = (words[-1] if len(words) else 0, tm[t, words[-1], c] if len(words) else 0)
            if len(words) > 1:
                tw[t, c, 0] = 0xFFFFFFFF
    nrem = np.zeros((D, R | 1), np.int32)
    nrem[:, :R] = n.T
    arrays = [np.ascontiguousarray(x) for x in (avail, lvl, lst, ent, tm, tw, slot_e, a, rec, nxt, np.arange(D, dtype=np.int32), nrem, np.array(lead, np.int32))]
    X, left, rounds = np.zeros((R, S), np.int32), np.zeros(S + 1, np.int32), np.zeros(1, np.int32)
    ptr = lambda x: x.ctypes.data_as(ctypes.c_void_p)
    auction.cta_reset()
    auction.cta_auction(lean, ptr(np.array([R, S, K, W, D, len(tiers), len(lead)], np.int32)), (ctypes.c_void_p * len(arrays))(*[x.ctypes.data for x in arrays]),
                        ptr(X), ptr(left), ptr(rounds))
    assert auction.cta_races() == 0, auction.cta_first().decode()
    assert auction.cta_stuck() == 0
    want = O.auction(R, D, K, n, np.where(tokens > 0, slot_e, -1), tokens, B, price_step=step)
    assert (X == want["X"]).all() and rounds[0] == want["rounds"]
    assert (left[:S] == np.where(tokens > 0, tokens - want["X"].sum(0), 0)).all()
