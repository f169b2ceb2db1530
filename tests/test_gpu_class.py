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
