"""Grouped contexts whose requests come in order are planned without a sort: at the edges of its tiles (1,792 requests)
and pieces (up to four tiles), with constants at the limits of its 32-bit arithmetic, and with the one request that
sends the call to the general path, against the oracle (whole numbers: bit for bit)."""
import numpy as np
import pytest

from oracle import oracle
from paper_2602_08747_b200 import binding as pb
from paper_2602_08747_b200 import inputs
from tests import util
from tests.gpu_util import assert_identical, run_library
from tests.test_kernel_variants_gpu import booked, several_ctx

pytestmark = pytest.mark.gpu

EDGES = [0, 1, 1791, 1792, 1793, 7167, 7168, 7169, 14_337, 40_000, 0, 30_000]


def check(wl, mode=pb.PARD_MODE_GROUPED):
    rc, got = run_library(wl, mode)
    assert rc == 0
    assert_identical(got, oracle.plan(wl.pipelines, wl.requests, wl.state, wl.n_ctx, 0))


@pytest.mark.parametrize("S", [1, 3, 4, 8, 9, 16, 17])
@pytest.mark.parametrize("span,B,m", [(3000, 2, 1), (40_000, 3, 7), (2_000_000_000, 4, 1), (10, 1, 1), (100_000, 2, 5000)])
def test_sizes_at_the_edges_of_tiles_and_pieces(S, span, B, m):
    check(several_ctx(len(EDGES), EDGES, seed=S, S=S, span=span, B=B, m=m))
    big = [16_384, 16_385, 65_536, 200_000]               # pieces of more than one tile from a million requests on
    if S == 8:
        check(several_ctx(20, big * 5, seed=7, S=S, span=span, B=B, m=m))


@pytest.mark.parametrize("S", [4, 16])
def test_one_queue_holds_nearly_all(S):
    wl = several_ctx(3, [20_000, 9_000, 30_000], S=S, span=50_000, m=30)
    wl.requests["stage"] = np.where(np.arange(wl.n) % 997 == 0, wl.requests["stage"], S - 1)
    check(wl)
    wl.requests["stage"] = 0
    check(wl)


@pytest.mark.parametrize("at", [1, 1791, 1792, 20_000, 38_999])
def test_one_deadline_steps_back(at):
    for S in (3, 8):
        wl = several_ctx(4, [20_000, 0, 9_000, 10_000], S=S)
        wl.requests["deadline_us"][at] = 0
        check(wl)


# ---- in order, but not for this path: the passes behind it then sort the stage bits alone ----------------------------
def radix_passes(wl):
    """The passes that a call's sort needed: word 3 of its workspace."""
    import torch

    pipes = [pb.pard_load_pipeline(p) for p in wl.pipelines]
    S = wl.state.stage_stride
    ws = pb.alloc_workspace(pb.pard_plan_workspace_bytes(wl.n, wl.n_ctx, S), "cuda")
    pb.pard_plan(pipes, pb.device_requests(wl.requests, "cuda"), wl.n, pb.device_state(wl.state, "cuda"), wl.n_ctx, pb.PARD_MODE_GROUPED,
                 pb.alloc_out(wl.n, wl.n_ctx * S, "cuda"), ws, stream=torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    for p in pipes:
        p.free()
    return int(ws[12:16].view(torch.int32).item())


def off_the_path(reason, n_ctx=3, per=20_000, **kw):
    wl = several_ctx(n_ctx, [per] * n_ctx, S=8, m=20, **kw)
    d = wl.requests["deadline_us"].reshape(n_ctx, per)
    if reason == "stage of 1 us":
        wl.pipelines = [util.pipeline(inputs.chain_edges(8), 8, [9, 30, 1, 7, 12, 5, 17, 8], bmax=4)]
    elif reason == "piece beyond 32 bits":
        d[1, per // 2:] += 1 << 32
    elif reason == "piece beyond 31 bits":
        d[n_ctx - 1, per // 3:] += 1 << 31
    elif reason == "booked long ago":
        d[0] += (1 << 31) + 5000
    return wl


@pytest.mark.parametrize("reason,n_ctx,per", [(r, c, k) for r in ("stage of 1 us", "piece beyond 32 bits", "piece beyond 31 bits", "booked long ago")
                                              for c, k in ((3, 20_000), (70, 16_384))] + [("stage of 1 us", 1025, 8_193)])
def test_in_order_for_the_passes_alone(reason, n_ctx, per):
    wl = off_the_path(reason, n_ctx, per)
    check(wl)
    assert radix_passes(wl) == 1
    for at in (per + 1, 2 * per - 1)[:1 if n_ctx > 1000 else 2]:                    # one step back, in the second ctx
        wl = off_the_path(reason, n_ctx, per)
        wl.requests["deadline_us"][at] = wl.requests["deadline_us"][at - 1] - 1
        check(wl)
        assert radix_passes(wl) > 1


@pytest.mark.parametrize("reason", ["", "stage of 1 us", "piece beyond 32 bits"])
@pytest.mark.parametrize("at", [1, 31, 32, 255, 256, 257, 1791, 1792, 1793, 2048, 20_001, 21_792, 39_999])
def test_no_step_back_is_missed(reason, at):
    """By one microsecond; behind a deadline too far ahead for 32-bit offsets, its low word small; and over several requests."""
    for far, until in ((0, at), (1 << 31, at), (1 << 32, at), ((1 << 32) - 5, at), (0, at + 300), (1 << 33, at + 300)):
        wl = off_the_path(reason)
        d = wl.requests["deadline_us"]
        if far:
            d[max(until - 300, at - 1):until] += far      # a step back at `until`
        elif until > at:
            d[at:until] -= 900                            # at `at` (and none behind)
        else:
            d[at] = d[at - 1] - 1
        check(wl)


@pytest.mark.parametrize("span", [3000, (1 << 31) - 3, (1 << 31) - 2, (1 << 31) - 1, 1 << 31, 1 << 33])
@pytest.mark.parametrize("d", [1, 7, (1 << 31) + 9, (1 << 32) + 9])
def test_constants_at_the_limits(span, d):
    targets = [0, 1, span, span + 2, (1 << 31) - 2, (1 << 31) - 1, 1 << 31, 1 << 40, -1, -(1 << 31), -(1 << 31) - 1]
    wl = booked(targets, span, d, n=8300)
    check(wl)
    for t in targets:                                     # without a ctx that the path does not take
        check(booked([t, t], span, d, n=8300))


def test_errors_are_still_reported():
    def rc(wl):
        return run_library(wl, pb.PARD_MODE_GROUPED, check=False)[0]

    for S in (4, 3):                                      # with passes inside the contexts, and without
        wl = several_ctx(3, [20_000, 9_000, 10_000], S=S)
        for field, value in (("stage", S), ("ctx", 3), ("deadline_us", -1), ("deadline_us", 1 << 60)):
            for at in (0, 25_000, wl.n - 1):
                bad = inputs.Workload("bad", wl.pipelines, wl.requests.copy(), wl.state, wl.n_ctx)
                bad.requests[field][at] = value
                assert rc(bad) == pb.PARD_EDATA, (field, at)
        check(wl)
    wl = several_ctx(3, [20_000, 9_000, 10_000], S=4)
    wl.requests["ctx"][100] = 1                           # not grouped
    assert rc(wl) == pb.PARD_EDATA
    wl = several_ctx(3, [20_000, 9_000, 10_000], S=4)
    wl.state.batch[1, 2] = 0                              # constants out of range, of an empty ctx and of one with requests
    for sizes in ([20_000, 0, 10_000], [20_000, 9_000, 10_000]):
        for sort in (True, False):
            assert rc(inputs.Workload("bad", wl.pipelines, several_ctx(3, sizes, S=4, sort=sort).requests, wl.state, 3)) == pb.PARD_EDATA
    wl = several_ctx(3, [20_000, 9_000, 10_000], S=4)
    short = util.pipeline(inputs.chain_edges(2), 2, [10, 20], bmax=4)     # a queue its pipeline lacks
    wl.pipelines = [wl.pipelines[0], short]
    wl.state.pipeline_of_ctx = np.array([0, 1, 0], np.int32)
    assert rc(wl) == pb.PARD_EDATA
    keep = ~((wl.requests["ctx"] == 1) & (wl.requests["stage"] >= 2))
    wl.requests = np.ascontiguousarray(wl.requests[keep])
    check(wl)


@pytest.mark.parametrize("ctx", [0, 1])
@pytest.mark.parametrize("crossing", [0, 1, 255, 256, 257, 600, 1039, 1040])
def test_deadlines_that_cross_the_limit_inside_the_last_piece(ctx, crossing):
    """Deadlines of a ctx one microsecond apart, the first one outside [0, 2^60) so many requests behind the beginning
    of the ctx's last piece (8,960: five tiles; 256 requests to a warp); 1,040: behind its last request."""
    wl = several_ctx(2, [10_000, 10_000], S=4, m=20)
    wl.state.now_us[ctx] = (1 << 60) - 20_000
    wl.requests["deadline_us"][10_000 * ctx:][:10_000] = (1 << 60) - 8_960 - crossing + np.arange(10_000)
    if crossing == 1040:
        check(wl)
        check(wl, 0)
    else:
        for mode in (pb.PARD_MODE_GROUPED, 0):
            assert run_library(wl, mode, check=False)[0] == pb.PARD_EDATA


@pytest.mark.parametrize("sizes", [[9000, 9000], [20_000, 0, 30_000], [65_536] * 20])
def test_wait_for_a_tile_runs_out_and_is_reported(sizes):
    wl = several_ctx(len(sizes), sizes, S=8, m=20)
    assert run_library(wl, pb.PARD_MODE_GROUPED | pb.PARD_MODE_TEST_STALL, check=False)[0] == pb.PARD_ETIMEOUT
    check(wl)


@pytest.mark.parametrize("shift", [0, 16])
@pytest.mark.parametrize("mode", [0, pb.PARD_MODE_GROUPED, pb.PARD_MODE_SCAN, pb.PARD_MODE_RAW, pb.PARD_MODE_FCFS])
@pytest.mark.parametrize("sizes", [[5000], [30_011], [3000, 7001], [20_000, 9_001]])
def test_outputs_on_16_byte_boundaries(shift, mode, sizes):
    """What the entry points ask of d_est_us and d_perm; the kernels' widest stores are of 32 bytes."""
    import torch

    for sort in (True, False):
        wl = several_ctx(len(sizes), sizes, S=4, m=9, sort=sort)
        want = oracle.plan(wl.pipelines, wl.requests, wl.state, wl.n_ctx, mode & (pb.PARD_MODE_RAW | pb.PARD_MODE_FCFS))
        pipes = [pb.pard_load_pipeline(p) for p in wl.pipelines]
        out = pb.alloc_out(wl.n, wl.n_ctx * 4, "cuda")
        out.est_us = torch.empty(wl.n + 4, dtype=torch.int64, device="cuda")[shift // 8:]
        out.perm = torch.empty(wl.n + 8, dtype=torch.int32, device="cuda")[shift // 4:]
        assert out.est_us.data_ptr() % 32 == shift and out.perm.data_ptr() % 32 == shift
        ws = pb.alloc_workspace(pb.pard_plan_workspace_bytes(wl.n, wl.n_ctx, 4), "cuda")
        pb.pard_plan_policy(pipes, pb.device_requests(wl.requests, "cuda"), None, wl.n, pb.device_state(wl.state, "cuda"), wl.n_ctx,
                            mode, out, ws, stream=torch.cuda.current_stream().cuda_stream)
        torch.cuda.synchronize()
        assert np.array_equal(out.est_us[:wl.n].cpu().numpy(), want["est_us"])
        assert np.array_equal(out.perm[:wl.n].cpu().numpy().view(np.uint32), want["perm"])
        for p in pipes:
            p.free()
