"""Dispatch metadata where a warp's span of a chunk is full, short or empty, with one and two rows of lane masks, with the counting
pass's counts kept and with spans counted again, against the oracle."""
import pytest
import torch

import oracle as O
import workloads as W
from helpers import cpu, make_planner, topology

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("E,K", [(64, 2), (640, 8)])                  # 81 and 705 bins: the latter with one row of masks
@pytest.mark.parametrize("seg", [1, 255, 257, 2047, 2048, 2052, 16383, 16384, 18441])
def test_dispatch_spans(seg, E, K):
    _check(8, seg, E, K)


@pytest.mark.parametrize("R,E,K,segs", [
    (8, 64, 2, (40, 41)), (8, 640, 8, (352, 353)),                    # 81 and 705 bins: half as many entries
    (128, 768, 8, (896, 897)),                                        # 1793 bins
    (128, 896, 8, (961, 15367, 15368)), (128, 1024, 8, (700, 16384, 16400))])         # 1921 and 2049: one scatter CTA per SM
def test_dispatch_counts_kept_or_counted_again(R, E, K, segs):
    for seg in segs:
        _check(R, seg, E, K)


def _check(R, seg, E, K):
    cfg = W.get_config("cfg1").replace(L=2, R=R, E=E, K=K, k=1, T=R * seg)
    e2r, _ = topology(cfg)
    pl = make_planner(cfg)
    g = torch.Generator(device="cuda").manual_seed(seg)
    new = (torch.rand((2, R * seg, 1), generator=g, device="cuda") ** 3 * (E + R * K)).int().clamp(0, E + R * K - 1)
    d = pl.dispatch(new)
    for l in range(2):
        want = O.dispatch(cpu(new)[l], cfg.R, E, K, e2r.numpy())
        for k in ("send_counts", "target_counts", "perm"):
            assert (cpu(d[k])[l] == want[k]).all()
        assert cpu(d["info"])[l] == 0
    pl.close()
