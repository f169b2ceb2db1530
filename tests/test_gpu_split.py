"""Phase 1 of few problems of at most 64 ranks (rows and columns in the registers of one or two warps): the edges of its builds (multiples of
four supply ranks, of eight demand ranks, and one more), ends on every iteration of a group of eight, folds, hand-backs, unaligned
blocks.  The sums are those of the lane grid that large batches take, so a batch of the same problems gives the same bits; and the
oracle."""
import pytest
import torch

from helpers import check_sinkhorn_problem, cpu

pytestmark = pytest.mark.gpu

SHAPES = [(3, ((1, 2), (2, 1))), (8, ((1, 7), (4, 4), (5, 3), (8, 8))), (17, ((4, 13), (8, 9), (9, 8), (16, 17))),
          (32, ((1, 31), (4, 16), (8, 24), (12, 17), (13, 8), (16, 25), (17, 15), (32, 32))), (33, ((8, 25), (9, 8), (33, 33))),
          (50, ((12, 38), (13, 33), (1, 49), (17, 32))), (64, ((8, 56), (16, 48), (15, 49), (20, 44), (21, 43), (24, 57), (25, 33), (32, 64), (40, 24)))]


@pytest.mark.parametrize("R,sizes", SHAPES)
@pytest.mark.parametrize("iters,tol,check_every", [(1, 0.0, 1), (8, 0.0, 1), (9, 1e-7, 1), (63, 0.0, 1), (300, 1e-4, 1), (300, 1e-4, 3), (90, 1e-9, 1)])
@pytest.mark.parametrize("eps", [0.05, 2.0])             # 0.05: drifts out of fp32's comfortable range, folds
def test_few_problems_as_a_batch_of_them_and_as_the_oracle(R, sizes, iters, tol, check_every, eps):
    import paper_2608_03676_b200 as P
    g = torch.Generator().manual_seed(100 * R + iters)
    C = 1.0 + 7.0 * torch.rand((R, R), generator=g)
    C.fill_diagonal_(0.0)
    n = len(sizes)
    s = torch.zeros((n, R)); d = torch.zeros((n, R))
    for b, (h, c) in enumerate(sizes):
        s[b, torch.randperm(R, generator=g)[:h]] = torch.randint(1, 4000, (h,), generator=g).float()
        free = torch.nonzero(s[b] == 0).ravel() if h + c <= R else torch.arange(R)
        d[b, free[:c]] = torch.randint(1, 900, (c,), generator=g).float()
        d[b] *= float(s[b].sum() / d[b].sum()) * (1.0 if b % 2 else 0.97)

    def solve(copies):
        pl = P.Planner(L=n * copies, R=R, E=R, K=1, k=1, T=R, e2r=torch.arange(R, dtype=torch.int32), C=C, eps=eps, max_iters=iters,
                       tol=tol, check_every=check_every)
        out = pl.sinkhorn(s.repeat(copies, 1).cuda(), d.repeat(copies, 1).cuda())
        out = {k: v.cpu() for k, v in out.items()}
        pl.close()
        return out

    sms = torch.cuda.get_device_properties(0).multi_processor_count
    few, more, batch = solve(1), solve(3 * sms // n), solve(4 * sms // n + 1)
    for name in ("plan", "iters", "row_err", "info"):
        want = batch[name][:n].contiguous().view(torch.int32)
        assert torch.equal(few[name].view(torch.int32), want), name
        assert torch.equal(more[name][-n:].contiguous().view(torch.int32), want), name
    if eps == 2.0 and check_every == 1:
        for b in range(n):
            check_sinkhorn_problem(s[b].numpy(), d[b].numpy(), C.numpy(), eps, cpu(few["plan"])[b], cpu(few["iters"])[b],
                                   cpu(few["row_err"])[b], iters, tol, check_every)
