"""What the host code queues, on a CPU with a fake runtime: streams, joins, errors, the kernels that a call takes."""
import ctypes

import pytest
import torch

import fake_cuda as F
import workloads as W


@pytest.fixture(scope="module")
def so(tmp_path_factory):
    return F.load(str(tmp_path_factory.mktemp("fake")))


def _host_planner(so, L=24):
    return F.FakePlanner(so, L, 16, 64, 2, 8, 16 * 1024, W.cost_matrix(16, 8, (0.0, 1.0, 10.0), None), tol=1e-6)


def _large_planner(so, R=256, L=12):                 # tables that taot_plan splits into layer groups
    return F.FakePlanner(so, L, R, 128, 1, 8, R * 2048, W.cost_matrix(R, 8, (0.0, 1.0, 6.0, 16.0), 4), tol=1e-6)


@pytest.mark.parametrize("make,call,groups", [(_host_planner, "plan_host_block", 6), (_large_planner, "plan", 6),
                                              (lambda so: _large_planner(so, 64, 24), "plan", 3)])
def test_a_failing_launch_leaves_nothing_behind_on_internal_streams(so, make, call, groups):
    """Whatever a call queued on streams of the handle is joined into the caller's stream, also when one of its launches or copies
    fails: the caller may free or reuse its buffers in the order of its own stream."""
    so.fake_reset()
    pl = make(so)
    assert getattr(pl, call)() == 0
    so.fake_reset()
    assert getattr(pl, call)() == 0
    whole = F.log(so)
    assert len({e.stream for e in whole if e.kind == F.LAUNCH}) >= groups and not F.not_joined(whole)
    for kind in (F.LAUNCH, F.COPY):
        for after in range(sum(e.kind == kind for e in whole)):
            so.fake_reset()
            so.fake_fail(kind, after)
            assert getattr(pl, call)() == -4
            assert not F.not_joined(F.log(so)), (kind, after)
            so.fake_reset()
            assert getattr(pl, call)() == 0 and [e.name for e in F.log(so)] == [e.name for e in whole]
    pl.close()


def _streams_of(so, pl):
    assert pl.plan_host_block() == 0
    return {e.stream for e in F.log(so) if e.kind in (F.LAUNCH, F.COPY)}


def test_streams_of_host_calls_are_made_when_a_host_call_is_in_sight(so):
    so.fake_reset()
    pl = _host_planner(so)
    assert not [e for e in F.log(so) if e.kind == F.STREAM_CREATE]
    assert pl.plan() == 0 and not [e for e in F.log(so) if e.kind == F.STREAM_CREATE]
    so.fake_reset()
    so.fake_capturing(1)                             # captured before any other host call: nothing is made, all on one stream
    assert _streams_of(so, pl) == {F.CALLER} and not [e for e in F.log(so) if e.kind in (F.STREAM_CREATE, F.EVENT_CREATE)]
    so.fake_reset()
    so.fake_fail(F.STREAM_CREATE, 2)
    assert pl.plan_host_block() == -4 and not F.not_joined(F.log(so))
    so.fake_reset()                                  # (what is there already is kept)
    assert len(_streams_of(so, pl)) == 6
    so.fake_reset()
    so.fake_capturing(1)
    assert len(_streams_of(so, pl)) == 6 and not [e for e in F.log(so) if e.kind in (F.STREAM_CREATE, F.EVENT_CREATE)]
    pl.close()
    pl = _host_planner(so)
    so.fake_reset()
    so.fake_fail(F.STREAM_CREATE, 0)
    assert pl.host_block_layout() == 0 and pl.host_block_layout() == 0
    so.fake_reset()
    assert len(_streams_of(so, pl)) == 6 and not [e for e in F.log(so) if e.kind in (F.STREAM_CREATE, F.EVENT_CREATE)]
    pl.close()


@pytest.mark.parametrize("cap,L,want", [("1", 24, 1), ("3", 24, 3), (None, 24, 6), (None, 5, 5), ("9", 7, 6)])
def test_the_cap_on_layer_groups_holds_for_host_calls(so, monkeypatch, cap, L, want):
    so.fake_reset()
    if cap:
        monkeypatch.setenv("TAOT_PLAN_GROUPS", cap)
    pl = _host_planner(so, L)
    assert len(_streams_of(so, pl)) == want and not F.not_joined(F.log(so))
    pl.close()


def _rough(R, seed=1):
    C = 1.0 + torch.rand((R, R), generator=torch.Generator().manual_seed(seed))
    C.fill_diagonal_(0.0)
    return C


@pytest.mark.parametrize("R", [4, 32, 64, 100, 256])
@pytest.mark.parametrize("general", [False, True])
def test_a_plan_releases_the_matching_kernel_only_behind_the_merge(so, R, general):
    """The matching kernel reads the merge's loads without waiting, so a kernel that releases it before its own wait needs another
    one in front that has waited for the merge."""
    so.fake_reset()
    so.fake_keep_arg(b"sinkhorn_kernel", ctypes.sizeof(F.SinkArgs))
    pl = F.FakePlanner(so, 3, R, 2 * R, 1, 2, 16 * R, _rough(R) if general else W.cost_matrix(R, 4, (0.0, 1.0, 8.0), None))
    assert pl.plan() == 0
    names = F.kernels(so)
    launches = [e for e in F.log(so) if e.kind == F.LAUNCH]
    at = names.index("sinkhorn_kernel")
    args = F.SinkArgs.from_buffer_copy(bytes(launches[at].arg))
    assert args.R == R and args.early == 1
    assert names[at - 1] not in ("merge_kernel", "hist_chunk_kernel") and names[at + 1] == "match_kernel"
    pl.close()


def _route(so, B, R, C, **kw):
    """Kernels of one Phase-1 call, in order, each named once."""
    so.fake_reset()
    pl = F.FakePlanner(so, B, R, R, 1, 1, R, C, **kw)
    so.fake_reset()
    assert pl.sinkhorn(B) == 0
    pl.close()
    return list(dict.fromkeys(F.kernels(so)))


@pytest.mark.parametrize("R,B,tol,want", [
    (32, 3, 0.0, ["sinkhorn_tile_kernel", "sinkhorn_kernel", "sinkhorn_input_guard_kernel"]),
    (64, 3, 1e-6, ["sinkhorn_tile_kernel", "sinkhorn_kernel", "sinkhorn_input_guard_kernel"]),
    (64, 3, 0.0, ["sinkhorn_class_kernel", "sinkhorn_kernel"]),
    (256, 300, 0.0, ["sinkhorn_class_kernel", "sinkhorn_kernel"]),
    (384, 300, 0.0, ["sinkhorn_class_tree_kernel", "sinkhorn_cluster_kernel"]),
    (1024, 3, 1e-6, ["sinkhorn_class_tree_kernel", "sinkhorn_cluster_kernel"])])
def test_kernels_of_phase_1_on_a_cost_with_classes(so, R, B, tol, want):
    assert _route(so, B, R, W.cost_matrix(R, 8, (0.0, 1.0, 6.0, 16.0), 4), tol=tol) == want


_WIDE = ["sinkhorn_wide_kernel", "sinkhorn_cluster_kernel", "sinkhorn_kernel", "sinkhorn_input_guard_kernel"]
_DENSE = ["tc_prepare_kernel", "sinkhorn_tc_halfstep_kernel", "tc_finalize_kernel", "tc_report_kernel", "sinkhorn_input_guard_kernel"]


@pytest.mark.parametrize("R,B,iters,tol,eps,want", [
    (512, 300, 63, 0.0, 1.0, _DENSE), (512, 300, 64, 0.0, 1.0, _WIDE), (512, 255, 63, 0.0, 1.0, _WIDE), (512, 300, 63, 1e-6, 1.0, _WIDE),
    (384, 300, 63, 0.0, 0.09, _WIDE), (300, 300, 63, 0.0, 1.0, _WIDE),             # C / eps beyond 20; no multiple of 128
    (640, 300, 500, 0.0, 1.0, _DENSE), (640, 255, 500, 0.0, 1.0, _WIDE[1:])])
def test_kernels_of_phase_1_on_a_cost_without_structure(so, R, B, iters, tol, eps, want):
    assert _route(so, B, R, _rough(R), tol=tol, max_iters=iters, eps=eps) == want


@pytest.mark.parametrize("R,L,iters,tol,made", [(512, 300, 63, 0.0, True), (640, 256, 500, 0.0, True), (512, 300, 64, 0.0, False),
                                                (640, 255, 500, 0.0, False), (640, 256, 500, 1e-6, False), (512, 3, 10, 0.0, False)])
def test_the_gibbs_kernel_is_made_only_for_handles_whose_calls_can_take_it(so, R, L, iters, tol, made):
    so.fake_reset()
    pl = F.FakePlanner(so, L, R, R, 1, 1, R, _rough(R), tol=tol, max_iters=iters)
    assert (16 * R * R in [e.obj for e in F.log(so) if e.kind == F.DEVICE_ALLOC]) == made
    pl.close()


@pytest.mark.parametrize("R,E,K,seg,kept", [(256, 1024, 8, 16384, False), (256, 1024, 8, 300, False), (64, 256, 2, 192, False),
                                            (64, 256, 2, 193, True), (128, 791, 8, 908, True), (128, 792, 8, 908, False), (128, 1023, 8, 16384, True)])
def test_dispatch_workspace_follows_the_entries_of_a_chunk(so, R, E, K, seg, kept):
    """Counts by warp take 16 bytes per bin and chunk; they are kept only where a chunk has entries enough for its bins."""
    pl = F.FakePlanner(so, 2, R, E, K, 1, R * seg, W.cost_matrix(R, 8, (0.0, 1.0, 6.0, 16.0), 4), max_iters=10)
    n = ctypes.c_size_t()
    assert so.taot_workspace_bytes(pl.handle, ctypes.byref(n)) == 0
    bins, S = E + R * K + 1, R * K
    rest = 4 * 2 * R * (2 * E + 4 + bins + 2 * E + min(E, S) + 1) + 256 * 2 * R + 2 * R * seg + 4096 * 16       # everything else, generously
    assert (n.value > 16 * bins * 2 * R) if kept else (n.value < rest)
    pl.close()


@pytest.mark.parametrize("far", [2.0, 8.0, 10.0])        # 10: with the price step of 0.1 some scores are equal
@pytest.mark.parametrize("R,E,K", [(2, 2, 1), (2, 5, 3), (3, 3, 1), (4, 4, 2), (8, 8, 1), (11, 2, 1), (16, 16, 1)])
def test_a_round_of_the_auction_reads_inside_its_shared_memory(so, R, E, K, far):
    """The arbiters [2][R + words of 32 ranks] lie behind 8 bytes an expert; a round of the general build reads those of eight words,
    33 apart, by 32 lanes, of either half."""
    so.fake_reset()
    pl = F.FakePlanner(so, 1, R, E, K, 1, R * 16, W.cost_matrix(R, 2, (0.0, 1.0, far), None))
    assert pl.plan() == 0
    smem = [e.obj for e in F.log(so) if e.kind == F.LAUNCH and e.name == b"match_kernel"]
    assert len(smem) == 1 and smem[0] >= 8 * E + 4 * (R + 1) + 4 * (7 * 33 + 32)
    pl.close()
