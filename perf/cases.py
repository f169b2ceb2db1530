"""Performance cases of the replica-placement planner: what a training or serving job asks of it, over the range of
sizes it is used at.

A case is one call (or the calls of one step) through the package's public entry points.  Kinds:
  plan      `Planner.plan`: routing table on the device -> loads, flow hint, placement, rewritten table
  host      `Planner.plan_host_block`: the same from pinned host memory back to pinned host memory
  dispatch  `Planner.dispatch`: send counts and send-buffer positions of a rewritten table
  sinkhorn  `Planner.sinkhorn`: Phase 1 alone on a batch of supply / demand vectors

Topologies are tiered (self / node / [rail group] / elsewhere) or "measured": the same tiers with every link's cost a few
per cent off its tier, as a job gets them that times its links.  Routing is Zipf-skewed over a permutation of the experts
that each layer draws anew, or sends a fraction of the tokens to the experts of one rank.
"""
import math

import torch

import paper_2608_03676_b200 as taot


# ---------------------------------------------------------------------------------------------------------------------
# the cases


def _plan(name, L, R, E, K, k, tokens, node, group, far, zipf_lo, zipf_hi, hot, eps_frac, iters, tol, kind="plan",
          cost="tiered", one_rank=False):
    """tokens: per source rank; node: ranks per node; group: nodes per rail group (0: no such tier); far: highest cost
    (1 inside a node); hot: fraction of the tokens whose last choice is one expert, or (one_rank) up to which fraction of
    the tokens goes to the experts of one rank; tol 0: exactly `iters` Sinkhorn iterations."""
    c = dict(kind=kind, L=L, R=R, E=E, K=K, k=k, tokens=tokens, node=node, group=group, far=far, zipf_lo=zipf_lo,
             zipf_hi=zipf_hi, hot=hot, eps_frac=eps_frac, iters=iters, tol=tol, cost=cost, one_rank=one_rank)
    if name:
        c["name"] = name
    return c


def _sinkhorn(name, B, R, node, group, far, eps_frac, iters, cost="tiered"):
    c = dict(kind="sinkhorn", B=B, R=R, node=node, group=group, far=far, eps_frac=eps_frac, iters=iters, cost=cost)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # one small layer, planned on the critical path of a step: nothing but latency and launches
        _plan("plan_8_ranks_1_layer", 1, 8, 32, 2, 2, 512, 4, 0, 8.0, 1.2, 1.2, 0.0, 0.05, 200, 0.0),
        # all layers of a two-node job at once; the table fits in L2
        _plan("plan_16_ranks", 24, 16, 64, 2, 8, 1024, 8, 0, 10.0, 1.0, 1.0, 0.0, 0.02, 1000, 1e-6),
        # the same step for a job whose router runs on the host side: pinned memory in and out
        _plan("host_16_ranks", 24, 16, 64, 2, 8, 1024, 8, 0, 10.0, 1.0, 1.0, 0.0, 0.02, 1000, 1e-6, kind="host"),
        # sizes that are no multiple of anything: 24 ranks, 1001 tokens each, top-6, three guest slots, measured link costs
        _plan("plan_24_ranks_ragged", 7, 24, 72, 3, 6, 1001, 8, 0, 4.0, 0.8, 1.4, 0.0, 0.05, 1000, 1e-6, cost="measured"),
        # 30 to 90 % of the tokens sent to one rank's experts: the sensitivity study's imbalance
        _plan("plan_32_ranks_one_hot_rank", 12, 32, 256, 2, 8, 2048, 8, 0, 3.0, 0.0, 0.0, 0.9, 1.0, 1000, 1e-6, one_rank=True),
        # a large training step: 58 layers, 1 GB of routing
        _plan("plan_64_ranks", 58, 64, 256, 2, 8, 8192, 8, 0, 12.0, 0.8, 1.4, 0.05, 0.01, 1000, 1e-6),
        # the largest: 256 ranks in rail groups, more ranks than experts, 1.6 GB of routing
        _plan("plan_256_ranks", 48, 256, 128, 1, 8, 4096, 8, 4, 16.0, 0.6, 1.6, 0.0, 0.005, 1000, 1e-6),
        # what the token all-to-all needs after the plan of the 58 layers
        _plan("dispatch_64_ranks", 58, 64, 256, 2, 8, 8192, 8, 0, 12.0, 0.8, 1.4, 0.05, 0.01, 200, 0.0, kind="dispatch"),
        # Phase 1 alone: one problem, a batch that fills the GPU, the largest topology, and measured link costs, where
        # nothing about the matrix can be used
        _sinkhorn("sinkhorn_64_ranks_1_problem", 1, 64, 8, 4, 16.0, 0.01, 500),
        _sinkhorn("sinkhorn_256_ranks_1024_problems", 1024, 256, 8, 4, 16.0, 0.1, 500),
        _sinkhorn("sinkhorn_1024_ranks_64_problems", 64, 1024, 8, 4, 16.0, 0.01, 500),
        _sinkhorn("sinkhorn_512_ranks_measured", 256, 512, 8, 4, 16.0, 0.1, 500, cost="measured"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case.  A drawn table is no larger than the largest listed one's, and a drawn solve does no more work than
    the largest listed solve."""
    u = rng.random()
    if u < 0.25:
        cost = "measured" if rng.random() < 0.3 else "tiered"
        node = rng.choice((4, 8, 8, 16))
        nodes = _log(rng, 2, 512 // node if cost == "measured" else 1024 // node)
        R = node * nodes if rng.random() < 0.7 else max(3, node * nodes - rng.randrange(node))
        most = (512 * 512 * 256 if cost == "measured" else 1024 * 1024 * 64) // (R * R)
        B = _log(rng, 1, max(1, min(4096, most)))
        return _sinkhorn(None, B, R, node, rng.choice((0, 2, 4)), rng.choice((8.0, 12.0, 16.0)),
                         rng.choice((0.1, 0.05, 0.02, 0.01)), rng.choice((100, 200, 500)), cost)
    kind = "plan" if u < 0.80 else ("dispatch" if u < 0.92 else "host")
    R = _log(rng, 4, 256)
    node = rng.choice((4, 8, 8))
    if rng.random() < 0.6:
        R = max(node, R // node * node)
    per = rng.choice((0.5, 1, 2, 4, 8)) if R >= 32 else rng.choice((1, 2, 4, 8))
    E = max(4, min(1024, int(R * per)))
    K = rng.choice((1, 2, 2, 3, 4))
    k = rng.choice((1, 2, 4, 6, 8))
    k = min(k, max(1, E // 2))
    L = _log(rng, 1, 60)
    tokens = _log(rng, 64, 8192)
    if rng.random() < 0.6:
        tokens = max(64, tokens // 64 * 64)
    most = 4_000_000 if kind == "host" else 400_000_000
    while L * R * tokens * k > most:
        if L > 8:
            L //= 2
        else:
            tokens = max(16, tokens // 2)
        if tokens == 16 and L <= 8:
            break
    one_rank = E // R >= k and rng.random() < 0.4
    fixed = rng.random() < 0.3
    return _plan(None, L, R, E, K, k, tokens, node, rng.choice((0, 0, 4)), rng.choice((3.0, 8.0, 12.0, 16.0)), 0.6, 1.6,
                 rng.choice((0.3, 0.6, 0.9)) if one_rank else rng.choice((0.0, 0.0, 0.05)),
                 rng.choice((0.01, 0.02, 0.05, 1.0)), 200 if fixed else 1000, 0.0 if fixed else 1e-6, kind=kind,
                 cost="measured" if rng.random() < 0.15 else "tiered", one_rank=one_rank)


# ---------------------------------------------------------------------------------------------------------------------
# inputs


def _topology(case):
    """Link costs [R, R]: 0 on the diagonal, 1 inside a node, then the rail group (if there is one) and the rest.  Part of
    the job, not of a step's inputs: the same for every seed."""
    R, node, far = case["R"], case["node"], float(case["far"])
    at = torch.arange(R) // node
    C = torch.full((R, R), far)
    if case["group"]:
        C[(at[:, None] // case["group"]) == (at[None, :] // case["group"])] = 0.375 * far
    C[at[:, None] == at[None, :]] = 1.0
    if case["cost"] == "measured":
        g = torch.Generator().manual_seed(977 * R + node)
        C = C * (1.0 + 0.05 * torch.rand((R, R), generator=g))
    C.fill_diagonal_(0.0)
    return C


def _home_ranks(case):
    """Experts spread evenly over the ranks, in order (fewer experts than ranks: every other rank hosts none)."""
    E, R = case["E"], case["R"]
    return (torch.arange(E) * R) // E


def _routing(case, seed):
    """Router output [L, T, k] int32 on the GPU: per layer a pool of tokens is routed (k distinct experts each, drawn
    without replacement by popularity) and the layer's tokens are taken from the pool at random."""
    L, E, k, T = case["L"], case["E"], case["k"], case["R"] * case["tokens"]
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    home = _home_ranks(case).cuda()
    out = torch.empty((L, T, k), dtype=torch.int32, device="cuda")
    pool = min(T, 16384)
    for l in range(L):
        u = torch.rand((3,), generator=g, device="cuda")
        if case["one_rank"]:
            share = case["hot"] * (1 + l % 3) / 3.0
            rank = (u[0] * case["R"]).long()
            logp = torch.zeros((pool, E), device="cuda")
            to_rank = torch.rand((pool, 1), generator=g, device="cuda") < share
            logp.masked_fill_(to_rank & (home != rank)[None, :], -1e30)
        else:
            s = case["zipf_lo"] + (case["zipf_hi"] - case["zipf_lo"]) * u[0]
            place = torch.randperm(E, generator=g, device="cuda").float()
            logp = -s * torch.log1p(place)[None, :]
        noise = torch.empty((pool, E), device="cuda").exponential_(generator=g)
        rows = torch.topk(logp - torch.log(noise), k, dim=1).indices
        if case["hot"] and not case["one_rank"]:
            hot = (u[1] * E).long().clamp_(max=E - 1)
            last = rows[:, k - 1]
            force = (torch.rand((pool,), generator=g, device="cuda") < case["hot"]) & ~(rows == hot).any(dim=1)
            rows[:, k - 1] = torch.where(force, hot, last)
        pick = torch.randint(0, pool, (T,), generator=g, device="cuda", dtype=torch.int32)
        torch.index_select(rows.int(), 0, pick, out=out[l])
    return out


def _rank_loads(B, R, seed):
    """Loads [B, R] of about 32768 tokens a rank, Zipf(1.2) over the ranks in an order of each problem's own."""
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    order = torch.argsort(torch.rand((B, R), generator=g, device="cuda"), dim=1)
    w = (order.double() + 1.0) ** -1.2
    w *= 1.0 + 0.02 * torch.rand((B, R), generator=g, device="cuda")
    return torch.round(w / w.sum(dim=1, keepdim=True) * (32768 * R)).int()


def _planner(case, **sizes):
    C = _topology(case)
    return taot.Planner(C=C, eps=float(case["eps_frac"]) * float(case["far"]), max_iters=case["iters"], **sizes)


def prepare(case, seed):
    if case["kind"] == "sinkhorn":
        B, R = case["B"], case["R"]
        pl = _planner(case, L=B, R=R, E=R, K=1, k=1, T=R, e2r=torch.arange(R))
        _, _, s, d = pl.excess_spare(_rank_loads(B, R, seed))
        out = dict(plan=torch.empty((B, R, R), device="cuda"), iters=torch.empty((B,), dtype=torch.int32, device="cuda"),
                   row_err=torch.empty((B,), device="cuda"), info=torch.zeros((B,), dtype=torch.int32, device="cuda"))
        return dict(kind="sinkhorn", planner=pl, s=s, d=d, out=out)
    pl = _planner(case, L=case["L"], R=case["R"], E=case["E"], K=case["K"], k=case["k"], T=case["R"] * case["tokens"],
                  e2r=_home_ranks(case), tol=case["tol"])
    table = _routing(case, seed)
    if case["kind"] == "host":
        return dict(kind="host", planner=pl, table=table.cpu().pin_memory(), out=pl.alloc_host_block())
    out = pl.alloc_outputs()
    if case["kind"] == "dispatch":
        new = pl.plan(table, out)["new_idx"].clone()
        del out, table
        return dict(kind="dispatch", planner=pl, table=new, out=pl.dispatch(new))
    return dict(kind="plan", planner=pl, table=table, out=out)


#: what a step acts on after a plan (the iteration and round counters and the status words are looked at now and then)
RESULTS = ("n", "expert_load", "rank_load", "excess", "spare", "plan", "slot_expert", "slot_tokens", "X", "new_idx")


def run(state):
    pl = state["planner"]
    if state["kind"] == "sinkhorn":
        out = pl.sinkhorn(state["s"], state["d"], out=state["out"])
        return dict(plan=out["plan"], iters=out["iters"])
    if state["kind"] == "dispatch":
        out = pl.dispatch(state["table"], out=state["out"])
        return dict(send_counts=out["send_counts"], target_counts=out["target_counts"], perm=out["perm"])
    if state["kind"] == "host":
        out = pl.plan_host_block(state["table"], state["out"])
    else:
        out = pl.plan(state["table"], out=state["out"])
    return {name: out[name] for name in RESULTS}


def work(case):
    R = case["R"]
    if case["kind"] == "sinkhorn":
        B = case["B"]
        # supply ranks x demand ranks of a Zipf load are about an eighth of the matrix; a tiered cost needs a few
        # operations per rank and half-step
        per_iter = 4 * R * R / 8 if case["cost"] == "measured" else 8 * R
        return {"bytes": B * (8 * R + 4 * R * R + 4), "flops": B * case["iters"] * per_iter}
    L, E, S, entries = case["L"], case["E"], R * case["K"], case["L"] * R * case["tokens"] * case["k"]
    if case["kind"] == "dispatch":
        return {"bytes": 8 * entries + 4 * L * R * (R + E + S), "flops": 0}
    return {"bytes": 8 * entries + 4 * L * (R * E + E + 3 * R + R * R + 2 * S + R * S), "flops": 0}


def tolerance(case):
    if case["kind"] == "dispatch":
        return "exact"
    if case["cost"] == "measured":          # 32-bit sums over all ranks, hundreds of times
        return {"rel": 5e-5, "max": 2e-4, "differ": 0.001}
    # 32-bit sums over hundreds of iterations, which two correct solves may stop one step apart; a placement score that
    # ties to the last bit of the plan may fall either way
    return {"rel": 2e-5, "max": 1e-4, "differ": 0.001}
