"""The merge of chunk counts with four experts a thread and one by one (expert counts that are no multiple of four), one and several
chunks a segment, groups of ranks that do not divide the CTA; and the reassignment on both sides of the number of chunks up to which
512 threads share one."""
import pytest
import torch

import oracle as O
import workloads as W
from helpers import cpu, make_planner, topology

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("R,E", [(1, 4), (3, 30), (8, 32), (33, 99), (33, 132), (7, 1024), (64, 1021), (256, 128), (256, 250)])
@pytest.mark.parametrize("seg", [5, 16384, 33000])
def test_merge_counts(R, E, seg):
    import paper_2608_03676_b200 as P
    L = 2
    e2r = (torch.arange(E) * R // E).int()
    C = W.cost_matrix(R, 4, (0.0, 1.0, 8.0), None)
    pl = P.Planner(L=L, R=R, E=E, K=1, k=1, T=R * seg, e2r=e2r, C=C, eps=1.0, max_iters=1)
    g = torch.Generator(device="cuda").manual_seed(R + E)
    idx = (torch.rand((L, R * seg, 1), generator=g, device="cuda") ** 2 * E).int().clamp_(0, E - 1)
    n, el, rl = [cpu(x) for x in pl.histogram(idx)[:3]]
    want = torch.zeros((L * R, E), dtype=torch.int64, device="cuda")
    want.scatter_add_(1, idx.view(L * R, seg).long(), torch.ones((L * R, seg), dtype=torch.int64, device="cuda"))
    want = cpu(want.view(L, R, E))
    assert (n.reshape(want.shape) == want).all() and (el.reshape(L, E) == want.sum(1)).all()
    rank = torch.zeros((L, R), dtype=torch.int64).index_add_(1, e2r.long(), torch.from_numpy(want.sum(1)))
    assert (rl.reshape(L, R) == rank.numpy()).all()
    _, _, s, d = pl.excess_spare(torch.from_numpy(rl).cuda())
    mean = rank.sum(1, keepdim=True) // R
    assert (cpu(s) == (rank - mean).clamp(min=0).float().numpy()).all() and (cpu(d) == (mean - rank).clamp(min=0).float().numpy()).all()
    pl.close()


@pytest.mark.parametrize("per,k", [(512, 8), (1013, 3)])              # staged as bytes; read in place
def test_reassignment_on_both_sides_of_the_line(per, k):
    line = 4 * torch.cuda.get_device_properties(0).multi_processor_count // 8
    base = W.get_config("cfg1").replace(L=line + 1, T=8 * per, k=k)
    e2r, _ = topology(base)
    g = torch.Generator().manual_seed(k)
    topk = torch.randint(0, base.E, (base.L, base.T, k), generator=g).int()
    topk[:, : base.T // 2] = topk[:, : base.T // 2] % 5                # skewed: splits in most chunks
    outs = []
    for L in (line, line + 1):
        pl = make_planner(base.replace(L=L))
        out = pl.plan(topk[:L].contiguous().cuda())
        outs.append({q: cpu(out[q]) for q in ("slot_expert", "X", "new_idx")})
        pl.close()
    for q in outs[0]:
        assert (outs[0][q] == outs[1][q][:line]).all()
    for l in (0, 1, line):
        o = outs[1]
        want = O.assign(topk[l].numpy(), base.R, base.E, base.K, o["slot_expert"][l].ravel(), o["X"][l])
        assert (o["new_idx"][l].reshape(-1) == want.reshape(-1)).all()
