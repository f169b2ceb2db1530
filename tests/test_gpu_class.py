"""Phase 1 on classes of interchangeable ranks (`taot_sinkhorn` with a fixed count beyond 32 ranks, any call beyond 256):
every build of the two kernels, at the edges of the class counts, with classes of unequal size, rows that cannot be written
16 bytes at a time, and batches on both sides of the launch rules, against the oracle."""
import numpy as np
import pytest
import torch

import oracle as O
import workloads as W
from helpers import check_sinkhorn_problem, cpu

pytestmark = pytest.mark.gpu


def _solve(C, B, eps, iters, tol=0.0, seed=3, shuffle=False):
    import paper_2608_03676_b200 as P
    R = C.shape[0]
    if shuffle:                                   # classes whose ranks are not neighbours
        p = torch.randperm(R, generator=torch.Generator().manual_seed(seed))
        C = C[p][:, p].contiguous()
    pl = P.Planner(L=B, R=R, E=R, K=1, k=1, T=R, e2r=torch.arange(R, dtype=torch.int32), C=C, eps=eps, max_iters=iters,
                   tol=tol)
    loads = W.sweep_rank_loads(B, R, seed=seed, device="cuda")
    ex, sp, s, d = pl.excess_spare(loads)
    out = pl.sinkhorn(s, d)
    again = pl.sinkhorn(s, d)
    torch.cuda.synchronize()
    assert torch.equal(out["plan"], again["plan"])
    plan, it, err, info = cpu(out["plan"]), cpu(out["iters"]), cpu(out["row_err"]), cpu(out["info"])
    assert ((info & ~(2 | 16)) == 0).all()
    for b in sorted({0, B // 2, B - 1}):
        check_sinkhorn_problem(cpu(s)[b], cpu(d)[b], C.numpy(), eps, plan[b], it[b], err[b], iters, tol)
    tot = s.double().sum(1)
    assert bool(((out["plan"].double().sum(1) - d.double()).abs().sum(1) <= 1e-5 * tot).all())
    pl.close()


@pytest.mark.parametrize("R,node", [(33, 33), (34, 17), (40, 20), (40, 10), (41, 9), (64, 8), (66, 4), (100, 4), (128, 4), (256, 8)])
@pytest.mark.parametrize("B", [1, 5])
def test_dense_builds_by_class_count(R, node, B):
    """1 to 32 nodes (the last one short where R is no multiple), three tiers."""
    _solve(W.cost_matrix(R, node, (0.0, 1.0, 6.0, 16.0), 2), B, 0.8, 41, shuffle=True)


@pytest.mark.parametrize("B", [295, 296, 303])
def test_dense_four_problems_per_block(B):
    _solve(W.cost_matrix(72, 8, (0.0, 1.0, 12.0), None), B, 0.12, 30)


def test_dense_with_any_cost_between_classes():
    """Nodes on a ring: the cost between two of them is their distance, not a tier."""
    n = torch.arange(120) // 8
    dist = (n[:, None] - n[None, :]).abs()
    C = 1.0 + 2.0 * torch.minimum(dist, 15 - dist).float()
    C.fill_diagonal_(0.0)
    _solve(C, 3, 0.7, 50)


@pytest.mark.parametrize("R,node,nodes_per_group,tiers", [
    (264, 8, 4, 3), (300, 8, 4, 3), (512, 8, 4, 3), (1024, 8, 4, 3),        # groups of 4, one per lane; a short last group
    (512, 8, 2, 3), (1020, 4, 4, 3),                                        # two groups per lane
    (1024, 4, 2, 3),                                                        # four
    (1024, 4, 8, 3),                                                        # groups of 8
    (400, 4, None, 2), (297, 9, None, 2)])                                  # no group tier
def test_tree_builds_by_hierarchy(R, node, nodes_per_group, tiers):
    C = W.cost_matrix(R, node, (0.0, 1.0, 6.0, 16.0)[:3 if tiers == 2 else 4], nodes_per_group)
    _solve(C, 2, 0.9, 33)


@pytest.mark.parametrize("R,B,eps,iters,tol", [(264, 300, 1.6, 20, 0.0), (512, 160, 1.9, 300, 1e-6), (384, 3, 0.05, 12, 0.0)])
def test_tree_batches_tolerance_and_costs_beyond_fp32(R, B, eps, iters, tol):
    """Four problems per block; the stopping rule; C / eps of 320, where iterates leave fp32 and are retaken in the log domain."""
    _solve(W.cost_matrix(R, 8, (0.0, 1.0, 6.0, 16.0), 4), B, eps, iters, tol)


def test_dense_cost_beyond_fp32():
    _solve(W.cost_matrix(64, 8, (0.0, 1.0, 12.0), None), 4, 0.012, 25)


@pytest.mark.parametrize("R,node,B,iters,tol,both", [
    (200, 8, 4, 30, 0.0, (1, 100)),           # up to 256 ranks: one rank with both, 100 x 200 (beyond the last kernel's shared memory)
    (256, 8, 2, 300, 1e-6, (1, 100)),         # (the tier sums hand back)
    (384, 8, 256, 30, 0.0, (1, 384, 200)),    # a batch that costs without classes solve as dense products
    (384, 8, 3, 25, 1e-3, (1, 384, 200)),
    (300, 4, 3, 40, 0.0, (300,)),
    (512, 8, 14, 20, 0.0, (1, 512)),          # clusters of the tree kernel hand back
    (1024, 8, 2, 12, 0.0, (1, 600))])
def test_ranks_with_supply_and_demand_are_handed_back_and_solved(R, node, B, iters, tol, both):
    """The class kernels take disjoint supports; problems with ranks in both (one, many, all) go to the kernels behind them,
    whatever the size of their matrix, and leave their neighbours alone."""
    import paper_2608_03676_b200 as P
    C = W.cost_matrix(R, node, (0.0, 1.0, 6.0, 16.0), 4)
    g = torch.Generator().manual_seed(R + B)
    pl = P.Planner(L=B, R=R, E=R, K=1, k=1, T=R, e2r=torch.arange(R, dtype=torch.int32), C=C, eps=1.6, max_iters=iters, tol=tol)
    ex, sp, s, d = (t.cpu() for t in pl.excess_spare(W.sweep_rank_loads(B, R, seed=5, device="cuda")))
    for b, n in enumerate(both):              # problems 0, 1, ...: the first n ranks of an order of their own have both
        p = torch.randperm(R, generator=g)[:n]
        if n == 1:
            s[b, p] += 100.0; d[b, p] += 50.0
        else:
            s[b].zero_(); d[b].zero_()
            s[b, p] = torch.randint(1, 900, (n,), generator=g).float()
            d[b, p] = torch.randint(1, 900, (n,), generator=g).float()
            if R <= 256:
                d[b] = torch.randint(1, 900, (R,), generator=g).float()
        d[b] *= 1.01 * float(s[b].sum() / d[b].sum())
    out = pl.sinkhorn(s.cuda(), d.cuda())
    torch.cuda.synchronize()
    info, it = cpu(out["info"]), cpu(out["iters"])
    assert ((info & ~2) == 0).all() and (it >= 1).all()
    for b in sorted({*range(len(both)), B - 1}):
        check_sinkhorn_problem(s[b].numpy(), d[b].numpy(), C.numpy(), 1.6, cpu(out["plan"])[b], it[b], cpu(out["row_err"])[b], iters, tol)
    pl.close()


def test_more_supply_ranks_than_the_tiles_hold_are_flagged_up_to_256_ranks():
    import paper_2608_03676_b200 as P
    R = 200
    pl = P.Planner(L=1, R=R, E=R, K=1, k=1, T=R, e2r=torch.arange(R, dtype=torch.int32), C=W.cost_matrix(R, 8, (0.0, 1.0, 6.0, 16.0), 4),
                   eps=1.6, max_iters=10)
    s = torch.ones((1, R), device="cuda"); d = torch.ones((1, R), device="cuda")
    s[0, :60] = 0.0                           # 140 x 200
    out = pl.sinkhorn(s, d)
    assert int(out["info"][0]) & P.INFO_SINKHORN_SIZE and float(out["plan"].abs().max()) == 0.0
    pl.close()
