"""Phase 1 with a cost without structure at 257 to 512 ranks (the kernel matrix in the registers of one CTA, rows beyond 64 in
its shared memory): the edges of its row builds (16, 32 and 64 supply ranks and one more; the largest products of supply and
demand ranks; few demand ranks), ragged rank counts, a fixed count and the stopping rule, against the oracle."""
import numpy as np
import pytest
import torch

from helpers import check_sinkhorn_problem, cpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("R,rows", [(257, (1, 16, 17, 32)), (288, (33, 64, 65, 2)), (300, (31, 63, 66, 15)), (512, (54, 64, 16, 200)),
                                    (257, (128, 250, 67, 256)), (301, (150, 185, 290, 68)), (512, (256, 288, 291, 285)), (511, (69, 448, 510, 130))])
@pytest.mark.parametrize("iters,tol,check_every", [(70, 0.0, 1), (300, 1e-5, 1), (300, 1e-5, 7)])
def test_wide_kernel_by_supply_ranks(R, rows, iters, tol, check_every):
    import paper_2608_03676_b200 as P
    g = torch.Generator().manual_seed(R)
    C = 1.0 + 15.0 * torch.rand((R, R), generator=g)
    C.fill_diagonal_(0.0)
    B, eps = len(rows), 2.0
    s = torch.zeros((B, R)); d = torch.zeros((B, R))
    for b, h in enumerate(rows):
        p = torch.randperm(R, generator=g)
        s[b, p[:h]] = torch.randint(1, 40000, (h,), generator=g).float()
        d[b, p[h:]] = torch.randint(1, 9000, (R - h,), generator=g).float()
        d[b] *= float(s[b].sum() / d[b].sum()) * (1.0 if b % 2 else 0.97)      # odd: enough room, even: the supply is scaled
    pl = P.Planner(L=B, R=R, E=R, K=1, k=1, T=R, e2r=torch.arange(R, dtype=torch.int32), C=C, eps=eps, max_iters=iters, tol=tol,
                   check_every=check_every)
    out = pl.sinkhorn(s.cuda(), d.cuda())
    torch.cuda.synchronize()
    for b in range(B):
        check_sinkhorn_problem(s[b].numpy(), d[b].numpy(), C.numpy(), eps, cpu(out["plan"])[b], cpu(out["iters"])[b],
                               cpu(out["row_err"])[b], iters, tol, check_every)
    pl.close()


@pytest.mark.parametrize("R,n", [(512, 512), (300, 180)])
def test_ranks_with_supply_and_demand_beyond_every_capacity(R, n):
    """All ranks (or 180 of 300) with both: the matrix is larger than a quarter of R x R, which disjoint supports never exceed."""
    import paper_2608_03676_b200 as P
    g = torch.Generator().manual_seed(R)
    C = 1.0 + 15.0 * torch.rand((R, R), generator=g)
    C.fill_diagonal_(0.0)
    s = torch.zeros((2, R)); d = torch.zeros((2, R))
    s[0, :n] = torch.randint(1, 900, (n,), generator=g).float(); d[0, R - n:] = torch.randint(1, 900, (n,), generator=g).float()
    s[1, :20] = 50.0; d[1, 20:] = 3.0
    pl = P.Planner(L=2, R=R, E=R, K=1, k=1, T=R, e2r=torch.arange(R, dtype=torch.int32), C=C, eps=2.0, max_iters=66)
    out = pl.sinkhorn(s.cuda(), d.cuda())
    assert ((cpu(out["info"]) & ~16) == 0).all()
    for b in range(2):
        check_sinkhorn_problem(s[b].numpy(), d[b].numpy(), C.numpy(), 2.0, cpu(out["plan"])[b], cpu(out["iters"])[b], cpu(out["row_err"])[b], 66, 0.0)
    pl.close()
