"""Phase 2 by one warp (at most 64 ranks, one or two per lane) and by the whole CTA, set up before Phase 1 has ended, against the oracle."""
import pytest

import oracle as O
import workloads as W
from helpers import cpu, make_planner, oracle_schedule_layer, topology

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("R,per_rank,K", [(2, 8, 2), (31, 5, 2), (32, 4, 3), (33, 8, 1), (63, 3, 4), (64, 12, 2), (65, 3, 2), (96, 6, 2)])
def test_matching_bit_exact(R, per_rank, K):
    cfg = W.get_config("cfg3").replace(L=3, R=R, E=R * per_rank, K=K, T=R * 450, gpus_per_node=4, max_iters=50, tol=0.0)
    e2r, C = topology(cfg)
    pl = make_planner(cfg)
    out = {k: cpu(v) for k, v in pl.plan(W.routing_topk(cfg, device="cuda")).items()}
    B = O.default_preference(C.numpy())
    for l in range(cfg.L):
        m, a = oracle_schedule_layer(cfg, e2r.numpy(), B, out["n"][l], out["expert_load"][l], out["rank_load"][l], out["plan"][l])
        assert (out["slot_expert"][l].ravel() == m["slot_expert"]).all()
        assert (out["X"][l] == a["X"]).all()
        assert out["rounds"][l].tolist() == [m["inner_rounds"], a["rounds"]]
    pl.close()
