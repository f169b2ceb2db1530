"""Phase 3 on classes of slots: one warp and several, the hand-over between them, word edges of the rank sets, remaining counts
in and out of shared memory, and pairs of equal score, against the oracle."""
import pytest
import torch

import oracle as O
import workloads as W
from helpers import cpu, make_planner, oracle_schedule_layer, topology

pytestmark = pytest.mark.gpu

BASE = W.get_config("cfg3").replace(L=2, max_iters=60, tol=0.0)
SHAPES = {
    "one_word": BASE.replace(R=32, E=128, T=32 * 512),
    "two_words_first_rank_of_the_second": BASE.replace(R=33, E=99, T=33 * 512),
    "three_words": BASE.replace(R=72, E=144, K=3, T=72 * 300),
    "many_classes": BASE.replace(R=120, E=480, K=3, T=120 * 700, gpus_per_node=4),       # more than 128 classes
    "counts_in_global_memory": BASE.replace(R=200, E=400, K=2, T=200 * 400),
    "eight_words_four_tiers": BASE.replace(R=256, E=256, K=2, T=256 * 300, tiers=(0.0, 1.0, 3.0, 9.0), nodes_per_group=4),
    "a_few_ranks": BASE.replace(R=2, E=6, K=1, T=2 * 999, k=2, gpus_per_node=1, tiers=(0.0, 1.0, 10.0)),
    "a_few_ranks_equal_scores": BASE.replace(R=4, E=8, K=2, T=4 * 999, k=2, gpus_per_node=2, tiers=(0.0, 1.0, 10.0)),
    "equal_scores": BASE.replace(R=48, E=192, K=2, T=48 * 600, tiers=(0.0, 1.0, 2.0)),   # bonus 1 and 0.5, step 0.125
}


@pytest.mark.parametrize("name", sorted(SHAPES))
@pytest.mark.parametrize("step,cap", [(0.1, 0), (0.125, 0), (0.1, 17), (1e-9, 0)])
def test_auction_bit_exact(name, step, cap):
    cfg = SHAPES[name]
    e2r, C = topology(cfg)
    topk = W.routing_topk(cfg, device="cuda")
    pl = make_planner(cfg, price_step=step, auction_max_rounds=cap)
    out = {k: cpu(v) for k, v in pl.plan(topk).items()}
    B = O.default_preference(C.numpy())
    for l in range(cfg.L):
        m, a = oracle_schedule_layer(cfg, e2r.numpy(), B, out["n"][l], out["expert_load"][l], out["rank_load"][l], out["plan"][l],
                                     price_step=step, auction_max_rounds=cap)
        assert (out["slot_expert"][l].ravel() == m["slot_expert"]).all()
        assert (out["X"][l] == a["X"]).all()
        assert out["rounds"][l].tolist() == [m["inner_rounds"], a["rounds"]]
        assert bool(out["info"][l] & 8) == (a["residual"] > 0)
    pl.close()


def _nested(R, levels):
    """Ranks in nested groups: the cost is that of the smallest group that holds both."""
    at = torch.arange(R)
    C = torch.full((R, R), 2.0 ** len(levels))
    for i, size in reversed(list(enumerate(levels))):
        C[(at[:, None] // size) == (at[None, :] // size)] = 2.0 ** i
    return C.fill_diagonal_(0.0)


def _check_nested(levels, R, E, K, step):
    import paper_2608_03676_b200 as P
    L, k = 2, 4
    C = _nested(R, levels)
    e2r = (torch.arange(E) * R // E).int()
    cfg = BASE.replace(L=L, R=R, E=E, K=K, k=k, T=R * 300)
    g = torch.Generator().manual_seed(E + len(levels))
    topk = torch.stack([torch.multinomial((1.0 + torch.randperm(E, generator=g)) ** -1.2, cfg.T * k, replacement=True, generator=g).view(cfg.T, k) for _ in range(L)]).int()
    pl = P.Planner(L=L, R=R, E=E, K=K, k=k, T=cfg.T, e2r=e2r, C=C, eps=0.5, max_iters=40, tol=0.0, price_step=step)
    out = {q: cpu(v) for q, v in pl.plan(topk.cuda()).items()}
    B = O.default_preference(C.numpy())
    for l in range(L):
        m, a = oracle_schedule_layer(cfg, e2r.numpy(), B, out["n"][l], out["expert_load"][l], out["rank_load"][l], out["plan"][l], price_step=step)
        assert (out["slot_expert"][l].ravel() == m["slot_expert"]).all()
        assert (out["X"][l] == a["X"]).all()
        assert out["rounds"][l].tolist() == [m["inner_rounds"], a["rounds"]]
    pl.close()


@pytest.mark.parametrize("levels,E", [((8, 16, 32, 64, 128), 128), ((8, 32, 64, 128), 256), ((4, 8, 16, 32, 64, 128), 100),
                                      ((2, 4, 8, 16, 32, 64, 128), 250), ((8, 64, 128), 1024)])
@pytest.mark.parametrize("step", [0.1, 0.125])
def test_one_slot_per_rank_with_tier_masks_in_global_memory(levels, E, step):
    """As many slots as ranks: the tier masks that find no room in shared memory go by host and not by class."""
    _check_nested(levels, 256, E, 1, step)


@pytest.mark.parametrize("levels,R,E", [((2, 4, 8, 16, 32), 64, 128), ((4, 8, 16, 32, 64, 128), 200, 100), ((2, 4, 8, 16, 32, 64, 128), 256, 250)])
def test_five_to_eight_tiers_with_two_slots_per_rank(levels, R, E):
    _check_nested(levels, R, E, 2, 0.1)
