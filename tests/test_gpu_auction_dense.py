"""Phase 3 by dense scan (measured costs: more bonus values than tiers): one to 32 lanes per slot, one and several passes, the
bonus matrix in and out of shared memory, win counts that tie, against the oracle."""
import pytest
import torch

import oracle as O
import workloads as W
from helpers import cpu, make_planner, oracle_schedule_layer, topology

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("R,per_rank,K", [(2, 8, 1), (8, 6, 2), (24, 3, 3), (33, 4, 1), (64, 4, 8), (120, 2, 2), (250, 2, 1)])
@pytest.mark.parametrize("step,cap", [(0.1, 0), (-0.05, 0), (0.1, 3)])
def test_dense_scan_bit_exact(R, per_rank, K, step, cap):
    import paper_2608_03676_b200 as P
    cfg = W.get_config("cfg3").replace(L=2, R=R, E=R * per_rank, K=K, T=R * 350, gpus_per_node=8, max_iters=40, tol=0.0)
    e2r, C = topology(cfg)
    g = torch.Generator().manual_seed(R)
    C = C * (1.0 + 0.2 * torch.rand(C.shape, generator=g))
    C.fill_diagonal_(0.0)
    pl = P.Planner(L=cfg.L, R=R, E=cfg.E, K=K, k=cfg.k, T=cfg.T, e2r=e2r, C=C, eps=cfg.eps, max_iters=40, tol=0.0, price_step=step,
                   auction_max_rounds=cap)
    out = {k: cpu(v) for k, v in pl.plan(W.routing_topk(cfg, device="cuda")).items()}
    B = O.default_preference(C.numpy())
    for l in range(cfg.L):
        m, a = oracle_schedule_layer(cfg, e2r.numpy(), B, out["n"][l], out["expert_load"][l], out["rank_load"][l], out["plan"][l],
                                     price_step=step, auction_max_rounds=cap)
        assert (out["slot_expert"][l].ravel() == m["slot_expert"]).all()
        assert (out["X"][l] == a["X"]).all()
        assert out["rounds"][l].tolist() == [m["inner_rounds"], a["rounds"]]
    pl.close()
