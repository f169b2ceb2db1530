"""Reassignment of chunks with many splits (one hot rank feeds most slots), from bytes, staged, and unaligned, against the oracle."""
import pytest
import torch

import oracle as O
import workloads as W
from helpers import cpu, make_planner, topology

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("R,E,K,per,k", [(32, 256, 2, 2048, 8), (32, 256, 4, 2560, 8), (16, 320, 8, 1500, 8), (24, 240, 6, 701, 5)])
def test_many_splits(R, E, K, per, k):
    cfg = W.get_config("cfg3").replace(L=2, R=R, E=E, K=K, k=k, T=R * per, gpus_per_node=8, max_iters=40, tol=0.0)
    e2r, _ = topology(cfg)
    hot = (e2r == 1).nonzero().flatten().int()
    g = torch.Generator().manual_seed(R + K)
    topk = torch.randint(0, E, (2, cfg.T, k), generator=g).int()
    pick = torch.rand(topk.shape, generator=g) < 0.6
    topk = torch.where(pick, hot[torch.randint(0, len(hot), topk.shape, generator=g)], topk).int().cuda()
    pl = make_planner(cfg)
    out = pl.plan(topk)
    for l in range(2):
        want = O.assign(cpu(topk)[l], R, E, K, cpu(out["slot_expert"])[l].ravel(), cpu(out["X"])[l])
        assert (cpu(out["new_idx"])[l].reshape(-1) == want.reshape(-1)).all()
    assert int((out["X"].reshape(2, R, -1) > 0).sum(2).max()) > 4
    pl.close()
