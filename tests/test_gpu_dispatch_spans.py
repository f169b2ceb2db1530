"""Dispatch metadata where a warp's span of a chunk is full, short or empty, with one and two rows of lane masks, against the oracle."""
import pytest
import torch

import oracle as O
import workloads as W
from helpers import cpu, make_planner, topology

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("E,K", [(64, 2), (640, 8)])                  # 81 and 705 bins: the latter with one row of masks
@pytest.mark.parametrize("seg", [1, 255, 257, 2047, 2048, 2052, 16383, 16384, 18441])
def test_dispatch_spans(seg, E, K):
    cfg = W.get_config("cfg1").replace(L=2, R=8, E=E, K=K, k=1, T=8 * seg)
    e2r, _ = topology(cfg)
    pl = make_planner(cfg)
    g = torch.Generator(device="cuda").manual_seed(seg)
    new = (torch.rand((2, 8 * seg, 1), generator=g, device="cuda") ** 3 * (E + 8 * K)).int().clamp(0, E + 8 * K - 1)
    d = pl.dispatch(new)
    for l in range(2):
        want = O.dispatch(cpu(new)[l], cfg.R, E, K, e2r.numpy())
        for k in ("send_counts", "target_counts", "perm"):
            assert (cpu(d[k])[l] == want[k]).all()
        assert cpu(d["info"])[l] == 0
    pl.close()
