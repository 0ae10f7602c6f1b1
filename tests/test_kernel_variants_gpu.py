"""The variants a dispatch chooses from, at the sizes where they can go wrong, against the oracle."""
import numpy as np
import pytest

from oracle import oracle
from paper_2602_08747_b200 import binding as pb
from paper_2602_08747_b200 import inputs
from tests import util
from tests.gpu_util import assert_identical, run_library

pytestmark = pytest.mark.gpu

FCFS, NEXUS = pb.PARD_MODE_FCFS, pb.PARD_MODE_NEXUS
RULES = pb.PARD_MODE_PATH_MASK | FCFS | NEXUS | pb.PARD_MODE_CLIPPER


def check(wl, mode=0):
    want = oracle.plan(wl.pipelines, wl.requests, wl.state, wl.n_ctx, mode & (RULES | pb.PARD_MODE_RAW))
    rc, got = run_library(wl, mode)
    assert rc == 0
    assert_identical(got, want)
    return got


def several_ctx(n_ctx, sizes, seed=0, S=3, span=3000, sort=True, mix=False, B=2, m=1):
    """Contexts of the given sizes on one chain; deadlines in order inside every ctx when `sort`."""
    rng = np.random.default_rng(seed)
    p = util.pipeline(inputs.chain_edges(S), S, list(rng.integers(5, 40, size=S)), bmax=max(B, 4))
    ctx = np.repeat(np.arange(n_ctx), sizes)
    d = 1000 + rng.integers(0, span, size=ctx.size)
    if sort:
        d = d[np.lexsort((d, ctx))]
    if mix:
        k = rng.permutation(ctx.size)
        ctx, d = ctx[k], d[k]
    st = util.state(n_ctx, S, inputs.n_slots(p), 1000, B, workers=m, w=rng.integers(0, 50, size=(n_ctx, inputs.n_slots(p))))
    return inputs.Workload("variants", [p], util.requests(d, rng.integers(0, S, size=ctx.size), ctx), st, n_ctx)


# ---- rounds closed by a warp, by a block, or 32 requests per step --------------------------------
@pytest.mark.parametrize("rule", [FCFS, NEXUS])
@pytest.mark.parametrize("cap", [63, 64, 65, 1000, 8191, 8193])
@pytest.mark.parametrize("n", [15, 2047, 2049, 8192, 8193, 30_011])
def test_walk_rounds_against_steps_and_queue_lengths(rule, cap, n):
    rng = np.random.default_rng(n + cap)
    p = util.pipeline([], 1, [13], bmax=4096)
    st = util.state(1, 1, 0, 0, cap // 2 if cap > 4096 else cap, workers=2 if cap > 4096 else 1)
    real = int(st.batch[0, 0] * st.workers[0, 0])
    for top in (1.0, 3.0):                                 # rounds the queue needs, and well beyond
        dl = rng.integers(0, int(13 * (n / real + 2) * top), size=n)
        if rule == NEXUS:                                  # mostly fitting, so that windows do fill
            dl[rng.random(n) < 0.999] = 10**6
        check(inputs.Workload("edge", [p], util.requests(dl), st, 1), rule)


# ---- a block per ctx, groups of eight positions against requests one by one --------------------------
@pytest.mark.parametrize("mode", [0, pb.PARD_MODE_RAW])
@pytest.mark.parametrize("m", [1, 2, 4, 40])                                  # batch rounds of 2, 4, 8 and 80
@pytest.mark.parametrize("sizes", [[767, 769, 5, 768, 0, 770], [2047, 2049, 3, 2048, 2051], [8191, 0, 1, 8192, 4100], [3001, 6, 0, 0, 7990]])
def test_groups_of_positions(sizes, m, mode):
    for S, sort, span in ((3, True, 40_000), (9, True, 3000), (16, False, 3000)):
        check(several_ctx(len(sizes), sizes, seed=m, S=S, sort=sort, m=m, span=span), mode | pb.PARD_MODE_GROUPED)
    check(several_ctx(1, [sizes[0]], seed=m, S=5, m=m, span=100), mode)       # one ctx, many equal deadlines


@pytest.mark.parametrize("mode", [0, pb.PARD_MODE_RAW])
@pytest.mark.parametrize("cap", [1, 3, 7, 8, 9, 15, 16])                      # a group's estimates one by one, or two of them
def test_groups_of_positions_across_batch_rounds(cap, mode):
    for sizes, S, span in (([2500, 8192, 1, 4099, 2049], 3, 6000), ([8191, 3001], 10, 300), ([2053] * 9, 1, 40_000)):
        for sort in (True, False):
            check(several_ctx(len(sizes), sizes, seed=cap, S=S, sort=sort, span=span, B=cap), mode | pb.PARD_MODE_GROUPED)


@pytest.mark.parametrize("mode", [0, pb.PARD_MODE_RAW])
@pytest.mark.parametrize("sizes", [[1023, 1024, 1025, 1], [2047, 2048, 2049, 0, 7], [1500] * 9, [8192, 8191, 3000], [1024], [1025], [2048], [2049]])
def test_windows_without_requests(sizes, mode):
    rng = np.random.default_rng(sum(sizes))
    for S, gap, expired in ((3, 0, 0.2), (3, 900, 0.0), (3, 900, 0.2), (8, 1500, 0.01), (3, 20_000, 0.1)):     # the last: more windows than the tables hold
        wl = several_ctx(len(sizes), sizes, seed=S, S=S, sort=False, span=3, m=2)
        kind = rng.random(wl.n)
        wl.requests["deadline_us"] += np.where(kind < expired, -900, np.where(kind < 0.6, gap, gap * 4 // 3 + 60))
        check(wl, mode | pb.PARD_MODE_GROUPED)                                # sorted by the block
        wl.requests = wl.requests[np.lexsort((wl.requests["deadline_us"], wl.requests["ctx"]))]
        check(wl, mode | pb.PARD_MODE_GROUPED)                                # in order


# ---- searched tables: entries of 16 queues in shared memory, or more than fit there --------------------
@pytest.mark.parametrize("mode", [0, pb.PARD_MODE_RAW])
@pytest.mark.parametrize("span", [2000, 5500, 9000, 40_000])                  # some 1,900 to 40,000 entries
def test_searched_tables_of_sixteen_queues(span, mode):
    for m in (1, 30):
        check(several_ctx(5, [1900, 1700, 0, 3000, 2001], S=16, sort=False, mix=True, span=span, m=m), mode)


def table_entries(wl, want):
    """Window-table entries of every queue: an end marker, and a window up to the last request's.  A queue's first request
    is estimated at A."""
    d = np.array([wl.pipelines[0].lat_us[o] for o in wl.pipelines[0].lat_offsets[:wl.state.stage_stride]])
    off, dl = want["seg_offsets"], wl.requests["deadline_us"][want["perm"]]
    out = np.zeros(off.size - 1, np.int64)
    for q in np.flatnonzero(np.diff(off)):
        X = int(dl[off[q]:off[q + 1]].max()) - int(want["est_us"][off[q]])
        out[q] = 1 if X < 0 else X // d[q % d.size] + 2
    return out


@pytest.mark.parametrize("mode", [0, pb.PARD_MODE_RAW])
@pytest.mark.parametrize("lo, hi", [(1500, 2500), (3850, 4096), (4097, 4350), (5500, 6500)])      # entries of a block's 16 queues; 4,096 fit
def test_searched_tables_within_the_workspace(lo, hi, mode):
    n_ctx, S, n = 5, 16, 900_000
    sizes = [200_000, 150_000, 0, 249_000, 301_000]
    for m in (1, 300):
        wl = several_ctx(n_ctx, sizes, S=S, sort=False, mix=True, span=1, m=m)
        d = wl.pipelines[0].lat_us[wl.pipelines[0].lat_offsets[:S]]
        want = oracle.plan(wl.pipelines, wl.requests, wl.state, n_ctx, mode)
        start = want["est_us"][want["seg_offsets"][:S]]                       # A of the first ctx's queues
        last = int(((lo + hi) / 2 - 1.5 * S + (start / d).sum()) / (1.0 / d).sum())
        wl.requests["deadline_us"] = np.random.default_rng(m).integers(1000, last + 1, size=n)
        want = oracle.plan(wl.pipelines, wl.requests, wl.state, n_ctx, mode)
        entries = table_entries(wl, want)
        blocks = entries.reshape(-1, 16).sum(axis=1)
        assert entries.sum() <= n // 32 + 4 * n_ctx * S + 1024                # all fit: nothing is left to the scan
        assert ((lo <= blocks[[0, 1, 3, 4]]) & (blocks[[0, 1, 3, 4]] <= hi)).all(), blocks
        rc, got = run_library(wl, mode)
        assert rc == 0
        assert_identical(got, want)
        wl.state.priority = np.zeros((n_ctx, S), np.uint8)                    # some queues without a table between the others
        wl.state.priority[:, ::3] = 1
        check(wl, mode)


# ---- mixed contexts: the origins of up to 64 in shared memory ------------------------------------------
@pytest.mark.parametrize("n_ctx, S", [(2, 20), (2, 40), (63, 1), (64, 1), (64, 3), (65, 3)])
def test_packing_of_mixed_contexts(n_ctx, S):
    rng = np.random.default_rng(n_ctx + S)
    sizes = np.bincount(rng.integers(0, n_ctx, size=20_001 + 70 * n_ctx), minlength=n_ctx)
    wl = several_ctx(n_ctx, sizes, S=S, sort=False, mix=True, m=3)
    wl.requests["deadline_us"] += (wl.requests["ctx"].astype(np.int64) % 7) << 33     # far apart: low words alone tell contexts' origins
    check(wl)
    wl.state.priority = (rng.random((n_ctx, S)) < 0.4).astype(np.uint8)
    check(wl)


@pytest.mark.parametrize("n_ctx, S", [(2, 20), (2, 40), (63, 1), (64, 1), (64, 3), (65, 3)])
def test_packing_of_mixed_contexts_far_apart(n_ctx, S):
    """Contexts whose clocks are far apart, each booked close to its own: every queue's constants stay short."""
    rng = np.random.default_rng(n_ctx + S)
    sizes = np.bincount(rng.integers(0, n_ctx, size=20_001 + 70 * n_ctx), minlength=n_ctx)
    wl = several_ctx(n_ctx, sizes, S=S, sort=False, mix=True, m=3)
    apart = ((np.arange(n_ctx, dtype=np.int64) * 5) % 7 << 33) + np.arange(n_ctx) * 1_000_003
    wl.requests["deadline_us"] += apart[wl.requests["ctx"]]
    wl.state.now_us += apart
    for mode in (0, pb.PARD_MODE_RAW):
        check(wl, mode)


# ---- arrival order, one pass straight from the requests: up to 256 queues -------------------------
@pytest.mark.parametrize("rule", [FCFS, NEXUS, FCFS | pb.PARD_MODE_PATH_MASK])
@pytest.mark.parametrize("queues", [2, 4, 5, 255, 256, 257])
@pytest.mark.parametrize("n", [8193, 24_575, 24_576, 60_001])
def test_arrival_order_from_the_requests(rule, queues, n):
    sizes = np.bincount(np.random.default_rng(n).integers(0, queues, size=n), minlength=queues)
    for S, far in ((1, 0), (1, 1 << 57)):                  # the last: offsets beyond the elements, looked up
        wl = several_ctx(queues, sizes, S=S, sort=False, mix=True, m=1 + n % 3)
        wl.requests["deadline_us"][::7] += far
        check(wl, rule)


@pytest.mark.parametrize("rule", [FCFS, NEXUS, FCFS | pb.PARD_MODE_PATH_MASK])
@pytest.mark.parametrize("n_ctx, S", [(1, 2), (85, 3), (64, 4), (32, 8), (8, 32), (4, 64)])       # 2, 255, 256 queues
@pytest.mark.parametrize("n", [8193, 24_576, 60_001])
def test_arrival_order_from_the_requests_of_several_stages(rule, n_ctx, S, n):
    rng = np.random.default_rng(n + S)
    sizes = np.bincount(rng.integers(0, n_ctx, size=n), minlength=n_ctx)
    for far in (0, 1 << 57):                               # the last: offsets beyond the elements, looked up
        wl = several_ctx(n_ctx, sizes, seed=n, S=S, sort=False, mix=True, m=1 + n % 3, span=40 * S + 3000)
        wl.requests["deadline_us"][::7] += far
        if rule & pb.PARD_MODE_PATH_MASK:                  # every stage but the last has one path
            wl.requests["flags"] = np.where(wl.requests["stage"] + 1 < S, rng.integers(0, 2, size=n), 0)
        check(wl, rule)


@pytest.mark.parametrize("rule", [FCFS, NEXUS, FCFS | pb.PARD_MODE_PATH_MASK, pb.PARD_MODE_CLIPPER])
@pytest.mark.parametrize("n, n_ctx", [(20_000, 2), (20_000, 64), (2_800_000, 64)])                # small tiles, wide ones
def test_errors_found_while_sorting_in_arrival_order(rule, n, n_ctx):
    """A request out of range is counted in the queue that its element is sorted into, and reported."""
    wl = several_ctx(n_ctx, np.full(n_ctx, n // n_ctx), S=4, sort=False, mix=True, m=5)
    wl.pipelines = [util.pipeline(inputs.chain_edges(3), 3, [20, 30, 7], bmax=4)]                 # (three of the row's four stages)
    wl.requests["stage"] %= 3
    wl.state.batch[:, 3] = 1
    n = wl.n
    good, arrivals = wl.requests.copy(), util.arrivals(np.full(n, 900), 500) if rule == pb.PARD_MODE_CLIPPER else None

    def status(change):
        wl.requests = good.copy()
        change(wl.requests)
        return run_library(wl, rule, check=False, arrivals=arrivals)[0]

    def put(field, at, value):
        def change(r):
            r[field][at] = value
        return change

    for at in (0, n // 2, n - 1, slice(100, n, 301)):
        for field, value in (("stage", 4), ("ctx", n_ctx), ("deadline_us", -5), ("deadline_us", 1 << 60)):
            assert status(put(field, at, value)) == pb.PARD_EDATA, (field, at)
    for ctx in (0, n_ctx // 2, n_ctx - 1):                 # a queue of a stage that the pipeline lacks; the last one is the last of all
        assert status(put("stage", int(np.flatnonzero(good["ctx"] == ctx)[5]), 3)) == pb.PARD_EDATA, ctx
    if n < 100_000:                                        # a wait between tiles runs out
        wl.requests = good
        assert run_library(wl, rule | pb.PARD_MODE_TEST_STALL, check=False, arrivals=arrivals)[0] == pb.PARD_ETIMEOUT
    wl.requests = good
    want = oracle.plan(wl.pipelines, good, wl.state, n_ctx, rule, arrivals)
    rc, got = run_library(wl, rule, arrivals=arrivals)     # the context still works afterwards
    assert rc == 0
    assert_identical(got, want)


@pytest.mark.parametrize("rule", [FCFS, NEXUS])
@pytest.mark.parametrize("n", [2_727_936, 2_727_937])      # the last size of the small tiles, the first of the wide ones
def test_arrival_order_from_the_requests_tiles(rule, n):
    check(several_ctx(2, [n // 3, n - n // 3], sort=False, mix=True, m=700, span=60_000), rule)


@pytest.mark.parametrize("sizes", [[5000, 0, 1, 4099], [200] * 40, [2100, 2048, 1]])
@pytest.mark.parametrize("mode", [FCFS, NEXUS, pb.PARD_MODE_PATH_MASK])
def test_walk_of_several_queues_with_heads_inside_tiles(sizes, mode):
    for m in (1, 40):
        check(several_ctx(len(sizes), sizes, sort=False, mix=True, m=m), mode)


# ---- requests that come in deadline order --------------------------------------------------------
@pytest.mark.parametrize("mode", [0, pb.PARD_MODE_GROUPED, pb.PARD_MODE_RAW, pb.PARD_MODE_SCAN])
@pytest.mark.parametrize("sizes", [[1], [8192], [8193], [20_011], [3000, 1, 0, 8192], [9000, 10_001, 8193, 8200]])
def test_requests_in_deadline_order(sizes, mode):
    if mode == pb.PARD_MODE_GROUPED and max(sizes) > 8192 >= sum(sizes) / len(sizes):
        pytest.skip("breaks the promise")
    wl = several_ctx(len(sizes), sizes, S=4, m=20)
    check(wl, mode)
    for at in (1, wl.n // 2, wl.n - 1):                    # in order but for one request
        if 0 < at < wl.n:
            w2 = several_ctx(len(sizes), sizes, S=4, m=20)
            w2.requests["deadline_us"][at] = 990
            check(w2, mode)
    wl.state.priority = np.ones((wl.n_ctx, 4), np.uint8)    # order of deadlines is not the queues' order then
    check(wl, mode)


def test_requests_in_deadline_order_across_mixed_contexts():
    wl = several_ctx(7, [3000] * 7, sort=False, mix=True)
    wl.requests["deadline_us"].sort()
    check(wl)
    wl.requests["deadline_us"][[5, 9000]] = wl.requests["deadline_us"][[9000, 5]]
    check(wl)


# ---- ranges of mixed contexts --------------------------------------------------------------------
@pytest.mark.parametrize("n_ctx,n", [(2, 3000), (500, 740_000), (4096, 9_000), (4097, 30_000)])
def test_ranges_of_contexts_in_mixed_order(n_ctx, n):
    rng = np.random.default_rng(n_ctx)
    wl = several_ctx(n_ctx, np.bincount(rng.integers(0, n_ctx, size=n), minlength=n_ctx), S=2, sort=False, mix=True, m=3)
    check(wl)
    wl.requests["deadline_us"][rng.integers(0, n, size=5)] += 1 << 33      # beyond 32-bit offsets from the first request
    check(wl)


# ---- batch-wait estimate: block shapes, ranks inside crowded and sparse bins, counters that wrap ---
@pytest.mark.parametrize("M", [1, 127, 2560, 2561, 5121, 10_240, 10_241, 20_481, 32_768])
def test_estimate_w_shapes(M):
    from tests.gpu_util import run_estimate_w
    rng = np.random.default_rng(M)
    wl = inputs.make("C2", n=10)
    S = wl.state.stage_stride
    for kind in range(3):
        s = (rng.integers(0, 1 << 24, size=(1, S, M)) if kind == 0 else np.full((1, S, M), 7) if kind == 1
             else rng.integers(0, 3, size=(1, S, M)) * 100_000)
        for num, den, seed in ((1, 10, 5), (0, 1, 2**64 - 1), (1, 1, 2**32 - 0x7F4A7C15 - 100_000)):
            want = oracle.estimate_w(wl.pipelines, None, 1, S, wl.state.slot_stride, s.astype(np.int32), num, den, seed)
            rc, got = run_estimate_w(wl, s.astype(np.int32), num, den, seed, fill=0)
            assert rc == 0
            assert np.array_equal(got, np.asarray(want).reshape(got.shape))


# ---- window tables of many queues, a warp for each: block and table edges ------------
@pytest.mark.parametrize("n_ctx,S,n", [(5, 15, 90_000), (5, 16, 90_000), (17, 16, 200_001), (1366, 3, 30_000), (4088, 1, 50_000),
                                       (511, 9, 20_000), (2731, 3, 1_100_000)])
@pytest.mark.parametrize("mode", [0, pb.PARD_MODE_RAW, pb.PARD_MODE_SCAN])
def test_window_tables_of_many_queues(n_ctx, S, n, mode):
    rng = np.random.default_rng(n)
    wl = several_ctx(n_ctx, np.bincount(rng.integers(0, n_ctx, size=n), minlength=n_ctx), S=S, sort=False, mix=True, m=2)
    check(wl, mode)
    wl.state.priority = rng.integers(0, 2, size=(n_ctx, S)).astype(np.uint8)
    check(wl, mode)


# ---- tiles of a small call: least size, last group of tiles, one and two rounds, beyond ----------------
@pytest.mark.parametrize("n", [8193, 2048 * 16, 2048 * 16 + 1, 2048 * 296, 2048 * 296 + 1, 296 * 4608, 296 * 4608 + 1,
                               2 * 296 * 4608, 2 * 296 * 4608 + 1])
def test_sort_tiles_at_the_edges_of_their_sizes(n):
    sizes = [n // 3, n // 7, n - n // 3 - n // 7]
    check(several_ctx(3, sizes, seed=n, sort=False, mix=True, span=3_000_000))


# ---- order check on low words: high words, contexts and single steps inside and between warps ----------
@pytest.mark.parametrize("at", [1, 31, 32, 33, 127, 128, 129, 5000, 19_999])
@pytest.mark.parametrize("kind", ["step back", "high word", "new ctx", "bad stage"])
def test_order_check_finds_the_single_step(at, kind):
    wl = several_ctx(2, [20_000, 0], span=10**6)
    if kind == "step back":
        wl.requests["deadline_us"][at] = wl.requests["deadline_us"][at - 1] - 1
    elif kind == "high word":                      # in order, low words stepping back
        wl.requests["deadline_us"][at:] += (1 << 32) - 10**6
    elif kind == "new ctx":
        wl.requests["ctx"][at:] = 1
        wl.requests["deadline_us"][at:] -= 900
    else:
        wl.requests["stage"][at] = 3
        assert run_library(wl, 0, check=False)[0] == pb.PARD_EDATA
        return
    check(wl)


# ---- packing with and without single words, queues' constants and counters of 32 bits ------------------
@pytest.mark.parametrize("span", [1 << 28, (1 << 29) - 1, 1 << 29, 1 << 31])
@pytest.mark.parametrize("n_ctx", [1, 3])
def test_packing_at_the_widths_of_its_words(span, n_ctx):
    wl = several_ctx(n_ctx, [40_000 // n_ctx] * n_ctx, sort=False, span=span)
    wl.requests["deadline_us"][:2] = 1000, 1000 + span
    for mode in (0, pb.PARD_MODE_GROUPED):
        check(wl, mode)


# ---- known paths: path sums at hand from 32 requests per queue on average on, else worked out by blocks ---
@pytest.mark.parametrize("off", [-1, 0, 1, 30_000])
@pytest.mark.parametrize("n_ctx", [1, 40])
def test_known_paths_with_sums_at_hand_and_without(off, n_ctx):
    from tests.test_policy_parity_gpu import draw_masks
    rng = np.random.default_rng(n_ctx)
    edges = [(0, 1), (0, 2), (1, 3), (2, 3), (3, 4), (3, 5)]      # the first stage has four paths
    p = util.pipeline(edges, 6, list(rng.integers(5, 40, size=6)), bmax=4)
    n = 32 * 6 * n_ctx + off
    st = util.state(n_ctx, 6, inputs.n_slots(p), 1000, 2, w=rng.integers(0, 50, size=(n_ctx, inputs.n_slots(p))))
    r = util.requests(1000 + rng.integers(0, 3000, size=n), rng.integers(0, 6, size=n), rng.integers(0, n_ctx, size=n))
    wl = inputs.Workload("paths", [p], r, st, n_ctx)
    draw_masks(wl, rng)
    check(wl, pb.PARD_MODE_PATH_MASK)


# ---- calls that run at the same time: every block waits for work in flight only, never for a block to be placed ---
@pytest.mark.parametrize("mode", [0, pb.PARD_MODE_SCAN])
def test_calls_at_the_same_time(mode):
    import torch
    works = [several_ctx(3, [450_000] * 3, seed=1, sort=False, mix=True, span=3_000_000),      # tiles fill the device: every pass in one kernel
             several_ctx(3, [430_001] * 3, seed=2, sort=False, mix=True, span=3_000_000),
             several_ctx(2, [1_400_000] * 2, seed=3, sort=False, mix=True, span=1 << 27),       # passes of their own, then the rest
             several_ctx(2, [700, 300], seed=4, sort=False, mix=True, span=1 << 20)]            # one tile
    calls = []
    for k, wl in enumerate(works):
        S = wl.state.stage_stride
        calls.append((wl, [pb.pard_load_pipeline(p) for p in wl.pipelines], pb.device_requests(wl.requests, "cuda:0"),
                      pb.device_state(wl.state, "cuda:0"), pb.alloc_out(wl.n, wl.n_ctx * S, "cuda:0"),
                      pb.alloc_workspace(pb.pard_plan_workspace_bytes(wl.n, wl.n_ctx, S), "cuda:0"),
                      torch.cuda.Stream(priority=-(k & 1))))
    torch.cuda.synchronize()
    for _ in range(8):
        for wl, pipes, req, state, out, ws, stream in calls:
            pb.pard_plan(pipes, req, wl.n, state, wl.n_ctx, mode | pb.PARD_MODE_NOWAIT, out, ws, stream=stream.cuda_stream)
    for wl, pipes, req, state, out, ws, stream in calls:
        assert pb.pard_plan_status(ws, stream=stream.cuda_stream) == 0
        got, want = pb.out_to_numpy(out, wl.n), oracle.plan(wl.pipelines, wl.requests, wl.state, wl.n_ctx)
        for key in ("seg_offsets", "perm", "keep", "est_us", "n_kept", "kept_idx", "seg_kept"):
            assert np.array_equal(got[key], want[key]), (wl.n, key)


def test_wait_between_the_passes_runs_out_and_is_reported():
    wl = several_ctx(2, [700, 300], sort=False, mix=True, span=1 << 20)      # one tile, several passes: no look-back to run out first
    rc, _ = run_library(wl, pb.PARD_MODE_TEST_STALL, check=False)
    assert rc == pb.PARD_ETIMEOUT
    check(wl)


# ---- requests found out of place by a block of a kernel whose other blocks are still starting ---------------------
@pytest.mark.parametrize("n_ctx,per", [(900, 2100), (40, 9000)])          # a block per ctx; passes inside the contexts' ranges
@pytest.mark.parametrize("at", [0, 0.3, 0.9])
def test_requests_out_of_place_while_blocks_start(n_ctx, per, at):
    wl = several_ctx(n_ctx, [per] * n_ctx, S=4, m=3)
    i, j = int(at * n_ctx) * per + per // 2 + 1, n_ctx * per - per // 2           # inside their contexts: the ranges look grouped
    wl.requests[[i, j]] = wl.requests[[j, i]]
    for _ in range(5):
        assert run_library(wl, pb.PARD_MODE_GROUPED, check=False)[0] == pb.PARD_EDATA
    check(wl)                                                             # legal without the promise
    wl.requests[[i, j]] = wl.requests[[j, i]]
    check(wl, pb.PARD_MODE_GROUPED)


# ---- out of order although grouped, decided by blocks that take one tile after the other: more tiles than blocks ------
@pytest.mark.parametrize("n", [5_304_320, 5_304_321, 6_500_001])           # 5,180 tiles of 1,024 on 148 multiprocessors, and more
def test_decision_behind_a_try_that_found_no_order(n):
    sizes = np.full(24, n // 24)
    sizes[7] += n - sizes.sum()
    check(several_ctx(24, sizes, S=4, sort=False, span=60_000, m=300), pb.PARD_MODE_GROUPED)


# ---- keys beyond 64 bits: a wait of the chunks' passes runs out, and nothing follows the half-sorted positions ------
@pytest.mark.parametrize("n", [1500, 10_000])                            # one tile, several
def test_wide_key_stops_behind_a_wait_that_ran_out(n):
    rng = np.random.default_rng(n)
    wl = several_ctx(300, np.bincount(rng.integers(0, 300, size=n), minlength=300), S=3, sort=False, mix=True)
    wl.requests["deadline_us"][:2] = 5, 1 << 59
    assert run_library(wl, pb.PARD_MODE_TEST_STALL, check=False)[0] == pb.PARD_ETIMEOUT
    check(wl)


# ---- queues booked far ahead (backlog) or long idle: 32-bit copies of A against the ctx's deadlines ------------------
def booked(targets, span, d, n=700, seed=0, grouped=True):
    """One ctx per target; in the last stage of each, A lies `target` us behind the ctx's smallest deadline."""
    rng = np.random.default_rng(seed)
    S, first = 3, 1 << 41
    p = util.pipeline(inputs.chain_edges(S), S, [11, 5, d], bmax=4)
    n_ctx = len(targets)
    ctx = np.repeat(np.arange(n_ctx), n)
    dl = first + rng.integers(0, span + 1, size=ctx.size)
    dl[::n], dl[n - 1::n] = first, first + span
    dl = dl[np.lexsort((dl, ctx))]
    if not grouped:
        k = rng.permutation(ctx.size)
        ctx, dl = ctx[k], dl[k]
    now = [min(first - 300, first + t - d) for t in targets]
    fa = np.zeros((n_ctx, S), np.int64)
    fa[:, S - 1] = [first + t - d for t in targets]
    st = util.state(n_ctx, S, inputs.n_slots(p), now, 2, free_at=fa, workers=3)
    return inputs.Workload("booked", [p], util.requests(dl, rng.integers(0, S, size=ctx.size), ctx), st, n_ctx)


@pytest.mark.parametrize("span", [0, 3000, (1 << 31) - 2, (1 << 31) - 1, 1 << 31])
@pytest.mark.parametrize("d", [7, 1 << 24])
def test_block_per_ctx_with_queues_booked_far_ahead(span, d):
    targets = [0, 1, span - 1, span, span + 1, span + 2, (1 << 31) - 2, (1 << 31) - 1, 1 << 31, (1 << 31) + 1, (1 << 32) + 5, 1 << 40,
               -1, -(1 << 31) + 1, -(1 << 31), -(1 << 31) - 1]
    for step_back in (False, True):                       # in deadline order, and sorted by the block
        wl = booked(targets, span, d)
        if step_back:
            wl.requests["deadline_us"][5::700] = wl.requests["deadline_us"][::700]
        for mode in (pb.PARD_MODE_GROUPED, pb.PARD_MODE_GROUPED | pb.PARD_MODE_RAW):
            check(wl, mode)
    for t in targets:
        check(booked([t], span, d))                       # a single ctx


@pytest.mark.parametrize("span", [3000, (1 << 29) - 1, 1 << 29, 1 << 31])
@pytest.mark.parametrize("d", [7, 1 << 24])
def test_single_words_with_queues_booked_far_ahead(span, d):
    targets = [0, span, span + 1, (1 << 29) - 1, 1 << 29, (1 << 29) + 1, (1 << 31) + 1, (1 << 32) + 5, 1 << 40,
               -1, -(1 << 29) + 1, -(1 << 29), -(1 << 29) - 1, -(1 << 31) - 1, -(1 << 32) - 5, -(1 << 40)]
    for grouped in (True, False):                        # one queue or several per thread of the decision
        wl = booked(targets, span, d, grouped=grouped)
        for mode in (0, pb.PARD_MODE_RAW, pb.PARD_MODE_SCAN):
            check(wl, mode)
        wl.state.priority = np.ones((wl.n_ctx, 3), np.uint8)              # A against the latest deadline
        for mode in (0, pb.PARD_MODE_RAW, pb.PARD_MODE_SCAN):
            check(wl, mode)
    for t in targets:                                    # few queues: tables counted while packing
        check(booked([t], span, d, n=9000))


# ---- a thread per queue: from 16,384 queues on, more than 128 of them per request of the average queue; 511 to a block ----
@pytest.mark.parametrize("n_ctx,S,n", [(16_383, 1, 60_000), (16_384, 1, 60_000), (16_384, 1, 2_097_151), (16_384, 1, 2_097_152),
                                       (511, 33, 30_000), (5462, 3, 1_100_000), (8193, 2, 9_000)])
@pytest.mark.parametrize("mode", [0, pb.PARD_MODE_RAW, pb.PARD_MODE_SCAN, FCFS])
def test_window_tables_of_very_many_queues(n_ctx, S, n, mode):
    rng = np.random.default_rng(n + S)
    wl = several_ctx(n_ctx, np.bincount(rng.integers(0, n_ctx, size=n), minlength=n_ctx), S=S, sort=False, mix=True, m=2)
    check(wl, mode)
    if mode != FCFS:
        wl.state.priority = rng.integers(0, 2, size=(n_ctx, S)).astype(np.uint8)
        check(wl, mode)


# ---- long queues walked by a cluster of eight blocks (131,072 requests a step), their rounds and their neighbours ------
@pytest.mark.parametrize("rule", [FCFS, NEXUS])
@pytest.mark.parametrize("cap", [16_383, 16_384, 65_535, 65_536, 131_072, 150_001])
@pytest.mark.parametrize("sizes", [[524_287], [524_288], [524_289, 5], [900_000, 0, 540_000, 560_000], [1_000_003]])
def test_walk_by_clusters(rule, cap, sizes):
    rng = np.random.default_rng(cap + len(sizes))
    p = util.pipeline([], 1, [13], bmax=4096)
    B = next(b for b in range(4096, 0, -1) if cap % b == 0)
    for share in (0.0, 0.00001, 0.3):                      # of late requests
        wl = several_ctx(len(sizes), sizes, S=1, sort=False)
        wl.pipelines = [p]
        wl.state = util.state(len(sizes), 1, 0, 0, B, workers=cap // B)
        late = rng.random(wl.n) < share
        wl.requests["deadline_us"] = np.where(late, rng.integers(0, 60, size=wl.n), 10**6)
        check(wl, rule)


@pytest.mark.parametrize("rule", [FCFS, NEXUS])
@pytest.mark.parametrize("walk", [0, pb.PARD_MODE_SCAN])   # by a cluster, by one block
def test_wait_for_copied_thresholds_runs_out_and_is_reported(rule, walk):
    wl = several_ctx(1, [600_001], S=1, sort=False)        # one queue in arrival order: no radix pass whose wait would run out first
    wl.pipelines = [util.pipeline([], 1, [13], bmax=4096)]
    wl.state = util.state(1, 1, 0, 0, 4096, workers=16)
    assert run_library(wl, rule | walk | pb.PARD_MODE_TEST_STALL, check=False)[0] == pb.PARD_ETIMEOUT
    check(wl, rule | walk)


# ---- the same where a cluster cannot be placed: by one block each (PARD_MODE_SCAN asks for it) -------------------------
@pytest.mark.parametrize("rule", [FCFS, NEXUS, pb.PARD_MODE_PATH_MASK])
@pytest.mark.parametrize("cap", [16_384, 65_536, 150_001])
@pytest.mark.parametrize("sizes", [[524_288], [900_000, 0, 540_000, 560_000]])
def test_walk_of_long_queues_without_clusters(rule, cap, sizes):
    B = next(b for b in range(4096, 0, -1) if cap % b == 0)
    wl = several_ctx(len(sizes), sizes, S=1, sort=False)
    rng = np.random.default_rng(cap)
    wl.pipelines = [util.pipeline([], 1, [13], bmax=4096)]
    wl.state = util.state(len(sizes), 1, 0, 0, B, workers=cap // B)
    wl.requests["deadline_us"] = np.where(rng.random(wl.n) < 0.001, rng.integers(0, 60, size=wl.n), 10**6)
    got = check(wl, rule | pb.PARD_MODE_SCAN)
    assert_identical(got, check(wl, rule))
