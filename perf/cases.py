"""The planner's work as its users have it done: what is timed, on which inputs, and how outputs compare.

Every case goes through the binding's public calls.  Inputs are drawn on the GPU from the seed; they
follow the shapes of the workloads in paper_2602_08747_b200/inputs.py (balanced variants: enough workers
that a sizeable share of the requests is kept)."""
from __future__ import annotations

import functools
import math
from types import SimpleNamespace

import numpy as np
import torch

from paper_2602_08747_b200 import binding as pb
from paper_2602_08747_b200 import inputs
from paper_2602_08747_b200 import replay as rp

DEV = "cuda"
NOW = inputs.NOW0
RULES = {"": 0, "known_paths": pb.PARD_MODE_PATH_MASK, "arrival_order": pb.PARD_MODE_FCFS,
         "nexus": pb.PARD_MODE_NEXUS, "clipper": pb.PARD_MODE_CLIPPER}
#: stages, batch sizes profiled, latency objectives in us (one is drawn per request), Zipf exponent of the queue depths
APPS = {"chain3": (3, 32, (150_000,), 0.0), "dag8": (8, 64, (300_000,), 1.2),
        "dag16": (16, 128, (700_000, 800_000, 1_000_000), 0.0), "sweep": (16, 128, (400_000,), 1.2)}
SWEEP_GRAPHS = 256          # different graphs in a what-if sweep
EPOCHS = 8                  # decision epochs of one replay
WINDOW_US = 5_000_000       # sliding window of the queueing delay
EPOCH_US = 600_000          # time between two epochs of a replay


# ---- the cases ------------------------------------------------------------------------------------
def plan(app, n_ctx, n, ragged=False, grouped=False, priority=False, wait=True, rule=""):
    return {"kind": "plan", "app": app, "n_ctx": n_ctx, "n": n, "ragged": ragged, "grouped": grouped,
            "priority": priority, "wait": wait, "rule": rule}


def host(app, n_ctx, n):
    return {"kind": "host", "app": app, "n_ctx": n_ctx, "n": n, "ragged": False}


def state(app, n_ctx, wait_samples, history, delay_samples):
    return {"kind": "state", "app": app, "n_ctx": n_ctx, "wait_samples": wait_samples, "history": history,
            "delay_samples": delay_samples}


def replay(app, n_ctx, n):
    return {"kind": "replay", "app": app, "n_ctx": n_ctx, "n": n, "ragged": False}


def listed():
    return [
        # a live broker deciding one small pipeline's queues: the caller waits for the decision
        dict(plan("chain3", 1, 3_001), name="live small"),
        # the same after a long overload: a million queued requests, Zipf queue depths
        dict(plan("dag8", 1, 1_000_003), name="live overloaded"),
        # the repository's headline workload: one snapshot of 2^24 requests, three objectives
        dict(plan("dag16", 1, 1 << 24, wait=False), name="snapshot large"),
        # many short epochs of different length in one call, as a capacity study sends them
        dict(plan("dag8", 96, 160_001, ragged=True, grouped=True), name="epochs few"),
        # a long bursty trace cut into epochs of equal length, all decided in one call
        dict(plan("dag8", 4_096, 4_096 * 8_192, grouped=True, wait=False), name="epochs many"),
        # what-if sweep: 256 different pipelines, each with its own queue
        dict(plan("sweep", 256, 256 * 65_536, grouped=True, wait=False), name="what-if sweep"),
        # many instances behind shared front ends: requests interleaved, some queues high budget first
        dict(plan("sweep", 512, 2_500_013, ragged=True, priority=True), name="instances interleaved"),
        # requests and results in (pinned) host memory: a broker without device buffers
        dict(host("dag8", 1, 300_007), name="host buffers"),
        # dynamic-path pipeline whose requests carry the path they will take
        dict(plan("dag16", 1, 1_000_003, rule="known_paths"), name="known paths"),
        # the Nexus rule over the large snapshot, as a comparison study runs it
        dict(plan("dag16", 1, 1 << 24, wait=False, rule="nexus"), name="nexus large"),
        # the State Planner's periodic refresh of w, q and the priorities for a sweep's instances
        dict(state("sweep", 256, 10_000, 600, 512), name="state refresh"),
        # closed-loop replay: eight epochs of 16 instances, queue state carried on the device
        dict(replay("sweep", 16, 1 << 20), name="replay"),
    ]


def draw(rng):
    def between(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    what = rng.choice(["live", "live", "snapshot", "few", "many", "sweep", "mixed", "host", "rule", "rule", "state", "replay"])
    if what == "live":
        return plan(rng.choice(["chain3", "dag8"]), 1, between(100, 1_500_000))
    if what == "snapshot":
        return plan("dag16", 1, between(1 << 18, 1 << 24), wait=rng.random() < 0.5)
    if what == "few":
        c = between(4, 500)
        return plan("dag8", c, c * between(200, 2_500) + rng.randrange(c), ragged=True, grouped=True)
    if what == "many":
        c = between(600, 4_096)
        return plan("dag8", c, c * between(256, 8_192), grouped=True, wait=False)
    if what == "sweep":
        c = between(24, 256)
        return plan("sweep", c, c * between(12_000, 65_536) + rng.randrange(c), ragged=True, grouped=True, wait=False)
    if what == "mixed":
        return plan("sweep", between(8, 1_024), between(1 << 16, 1 << 22), ragged=True, priority=rng.random() < 0.7)
    if what == "host":
        return host("dag8", between(1, 64), between(4_000, 1 << 22))
    if what == "rule":
        c = between(1, 64)
        return plan(rng.choice(["dag8", "dag16"]), c, between(1 << 16, 1 << 23), ragged=c > 1,
                    rule=rng.choice([r for r in RULES if r]))
    if what == "state":
        return state("sweep", between(1, 256), between(500, 20_000), between(20, 2_000), between(32, 2_048))
    return replay("sweep", between(1, 64), between(1 << 13, 1 << 20))


# ---- inputs ---------------------------------------------------------------------------------------
@functools.lru_cache(maxsize=None)
def graphs(app):
    """Edges and number of stages of the pipelines; a sweep has many, the other applications one."""
    if app != "sweep":
        return ((APPS[app][0], {"chain3": inputs.chain_edges(3), "dag8": inputs.DAG8_EDGES, "dag16": inputs.DAG16_EDGES}[app]),)
    rng = np.random.default_rng(4)
    sizes = [int(s) for s in rng.integers(4, 17, size=SWEEP_GRAPHS)]
    return tuple((s, inputs.random_dag_edges(rng, s)) for s in sizes)


@functools.lru_cache(maxsize=None)
def slots(app):
    """Per graph, the lengths of the downstream paths of all its (stage, path) slots."""
    out = []
    for n_stages, edges in graphs(app):
        succ = [[b for a, b in edges if a == k] for k in range(n_stages)]

        @functools.lru_cache(maxsize=None)
        def lengths(k):
            return [1] if not succ[k] else [1 + m for j in succ[k] for m in lengths(j)]

        out.append([m for k in range(n_stages) for j in succ[k] for m in lengths(j)])
    return out


def pipelines_used(case):
    return min(case["n_ctx"], len(graphs(case["app"])))


def deployment(case, seed):
    """Loaded pipelines and the queue state around them (host arrays)."""
    rng = np.random.default_rng(seed)
    app, n_ctx = case["app"], case["n_ctx"]
    S, bmax, slo, _ = APPS[app]
    P = pipelines_used(case)
    R = max(len(s) for s in slots(app))
    n_stages = np.array([g[0] for g in graphs(app)[:P]])
    base, slope = rng.integers(2000, 8001, size=(P, S, 1)), rng.integers(200, 1501, size=(P, S, bmax))
    if app != "dag16":                       # linear profiles; the 16-stage application has a slope per batch size
        slope[:] = slope[:, :, :1]
    lat = base + np.cumsum(slope, axis=2)
    pipes = [inputs.make_pipeline(edges, s, [bmax] * s, lat[i, :s]) for i, (s, edges) in enumerate(graphs(app)[:P])]
    of_ctx = (np.arange(n_ctx) % P).astype(np.int32)
    there = np.arange(S)[None, :] < n_stages[of_ctx][:, None]
    batch = np.where(there, rng.integers(bmax // 4, bmax + 1, size=(n_ctx, S)), 1).astype(np.int32)
    d = np.where(there, lat[of_ctx[:, None], np.arange(S)[None, :], batch - 1], 1)
    now = NOW + rng.integers(0, 1_000_000, size=n_ctx)
    st = inputs.QueueState(S, R, now, batch, now[:, None] + rng.integers(0, d), rng.integers(0, d + 1),
                           rng.integers(0, (0.31 * d.sum(axis=1)).astype(np.int64)[:, None] + 1, size=(n_ctx, R)),
                           None, of_ctx if P > 1 else None)
    if case.get("priority"):
        st.priority = (rng.random((n_ctx, S)) < 0.3).astype(np.uint8)
    return SimpleNamespace(pipes=[pb.pard_load_pipeline(p) for p in pipes], st=st, d=d, n_stages=n_stages[of_ctx])


def requests(case, dep, seed, now):
    """Requests of all contexts at the instants `now`: [n, 2] int64 = the 16-byte records, and their queues' sizes."""
    app, n, n_ctx = case["app"], case["n"], case["n_ctx"]
    S, _, slos, zipf = APPS[app]
    rng = np.random.default_rng(seed + 1)
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)

    def uniform(shape=n):
        return torch.rand(shape, generator=g, device=DEV, dtype=torch.float64)

    share = 0.5 + rng.random(n_ctx) if case["ragged"] else np.ones(n_ctx)
    sizes = np.floor(n * share / share.sum()).astype(np.int64)
    sizes[:n - int(sizes.sum())] += 1
    first = np.concatenate([[0], np.cumsum(sizes)[:-1]])
    ctx = torch.repeat_interleave(torch.arange(n_ctx, device=DEV), torch.from_numpy(sizes).to(DEV), output_size=n)
    # queues: Zipf weights over a random order of the context's stages
    rank = np.argsort(np.where(np.arange(S)[None, :] < dep.n_stages[:, None], rng.random((n_ctx, S)), 2.0), axis=1)
    weight = np.where(np.arange(S)[None, :] < dep.n_stages[:, None], (np.arange(S) + 1.0) ** -zipf, 0.0)
    cdf = np.minimum(np.cumsum(weight, axis=1) / weight.sum(axis=1, keepdims=True), 1.0)
    steps = torch.from_numpy((np.arange(n_ctx)[:, None] + cdf).reshape(-1)).to(DEV)
    at = torch.searchsorted(steps, ctx + uniform().clamp_(max=1 - 1e-9), right=True) - ctx * S
    at = torch.minimum(at.clamp_(min=0), torch.from_numpy(dep.n_stages).to(DEV)[ctx] - 1)
    stage = torch.from_numpy(rank.reshape(-1)).to(DEV)[ctx * S + at]
    # arrivals before `now`: uniform over the last fraction of a second, or a Poisson stream of 50k requests/s with bursts ten times as dense
    now_of = torch.from_numpy(now).to(DEV)[ctx]
    if zipf:
        gap = torch.from_numpy(np.where(rng.random(n_ctx) < 0.2, 2.0, 20.0)).to(DEV)[ctx]
        t = torch.cumsum(-gap * torch.log1p(-uniform()), 0)
        last = torch.from_numpy(first + sizes - 1).to(DEV).clamp_(min=0)
        arrive = now_of - (t[last][ctx] - t).to(torch.int64)
    else:
        arrive = now_of - (uniform() * min(400_000, slos[0] * 4 // 3)).to(torch.int64)
    slo = torch.tensor(slos, device=DEV)[torch.randint(len(slos), (n,), generator=g, device=DEV)]
    flags = torch.zeros_like(ctx)
    if case.get("rule") == "known_paths":    # unknown, the first path, or one of the first two
        flags = torch.tensor([0, 1, 3], device=DEV)[torch.randint(3, (n,), generator=g, device=DEV)]
    rec = torch.stack([arrive + slo, ctx | (stage << 32) | (flags << 48)], dim=1)
    arrivals = torch.stack([arrive, slo], dim=1)
    if n_ctx > 1 and not case.get("grouped") and case["kind"] != "replay":     # a replay's epochs come instance by instance
        mix = torch.randperm(n, generator=g, device=DEV)
        rec, arrivals = rec[mix], arrivals[mix]
    depth = torch.bincount(ctx * S + stage, minlength=n_ctx * S).reshape(n_ctx, S).cpu().numpy()
    return rec.contiguous(), arrivals.contiguous(), depth


def balance(dep, depth, slos):
    """Workers such that a queue drains in about half an objective."""
    half = int(np.mean(slos)) // 2
    dep.st.workers = np.maximum(1, -(-depth * dep.d // (dep.st.batch.astype(np.int64) * half))).astype(np.int32)


def prepare(case, seed):
    dep = deployment(case, seed)
    st, app = dep.st, case["app"]
    S, R, n_ctx = st.stage_stride, st.slot_stride, case["n_ctx"]
    s = SimpleNamespace(case=case, pipes=dep.pipes, S=S, R=R, n_ctx=n_ctx, stream=torch.cuda.current_stream().cuda_stream)
    if case["kind"] == "state":
        return prepare_state(case, dep, seed, s)
    s.n = case["n"]
    rec, arrivals, depth = requests(case, dep, seed, st.now_us)
    balance(dep, depth, APPS[app][2])
    if case["kind"] == "replay":
        s.now = torch.from_numpy(np.stack([st.now_us + e * EPOCH_US for e in range(EPOCHS)])).to(DEV)
        s.req = [rec.view(torch.uint8)] + [requests(case, dep, seed + 1000 * e, st.now_us + e * EPOCH_US)[0].view(torch.uint8)
                                           for e in range(1, EPOCHS)]
        s.replay = rp.Replay(s.pipes, st.pipeline_of_ctx, n_ctx, S, R, st.batch, st.workers, st.free_at_us, st.w_us,
                             None, 64, WINDOW_US, s.n, DEV)
        s.free_at = s.replay.state.free_at_us.clone()
        s.total, s.kept = (torch.zeros((EPOCHS, n_ctx), dtype=torch.int64, device=DEV) for _ in range(2))
        return s
    if case["kind"] == "host":
        def pin(a):
            return None if a is None else torch.from_numpy(np.ascontiguousarray(a)).pin_memory()

        s.req = rec.view(torch.uint8).cpu().pin_memory()
        s.state = pb.QueueStateArrays(S, R, pin(st.now_us), pin(st.batch), pin(st.free_at_us), pin(st.q_us), pin(st.w_us),
                                      pin(st.workers), pin(st.pipeline_of_ctx))
        out = pb.alloc_out(s.n, n_ctx * S, "cpu")
        s.out = pb.PlanOut(**{k: v.zero_().pin_memory() for k, v in vars(out).items()})
        s.ws = pb.alloc_workspace(pb.pard_plan_host_workspace_bytes(s.n, n_ctx, S, R), DEV)
        return s
    s.req = rec.view(torch.uint8)
    s.arrivals = arrivals.view(torch.uint8) if case["rule"] == "clipper" else None
    s.mode = RULES[case["rule"]] | (pb.PARD_MODE_GROUPED if case["grouped"] else 0) | (0 if case["wait"] else pb.PARD_MODE_NOWAIT)
    s.state = pb.device_state(st, DEV)
    s.out = pb.alloc_out(s.n, n_ctx * S, DEV)
    s.out.kept_idx.zero_()                   # a call writes its first n_kept entries
    s.ws = pb.alloc_workspace(pb.pard_plan_workspace_bytes(s.n, n_ctx, S), DEV)
    s.total, s.kept = (torch.empty(n_ctx, dtype=torch.int64, device=DEV) for _ in range(2))
    return s


def prepare_state(case, dep, seed, s):
    st, n_ctx, S = dep.st, s.n_ctx, s.S
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    d = torch.from_numpy(dep.d).to(DEV)[:, :, None]

    def fraction(m):
        return torch.rand((n_ctx, S, m), generator=g, device=DEV)

    st.workers = np.random.default_rng(seed + 2).integers(1, 9, size=st.batch.shape).astype(np.int32)
    s.state = pb.device_state(st, DEV)
    s.waits = (fraction(case["wait_samples"]) * d).to(torch.int32)
    # arrivals per 100 ms around the modules' throughput
    mean = (s.state.batch * s.state.workers)[:, :, None] * 100_000.0 / d
    s.history = (mean * (0.3 + 1.4 * fraction(case["history"]))).to(torch.int32)
    # delays recorded over the last eight seconds, a tenth of the slots still empty
    age = (fraction(case["delay_samples"]) * 8_000_000).to(torch.int64)
    s.delay_time = torch.where(fraction(case["delay_samples"]) < 0.1, -1, s.state.now_us[:, None, None] - age)
    s.delay = (fraction(case["delay_samples"]) * 2 * d).to(torch.int32)
    s.w = torch.zeros((n_ctx, s.R), dtype=torch.int64, device=DEV)
    s.q = torch.zeros((n_ctx, S), dtype=torch.int64, device=DEV)
    s.priority = torch.zeros((n_ctx, S), dtype=torch.uint8, device=DEV)
    s.ws_w = pb.alloc_workspace(pb.pard_estimate_w_workspace_bytes(len(s.pipes)), DEV)
    s.ws_q = pb.alloc_workspace(pb.pard_update_queue_delay_workspace_bytes(), DEV)
    s.ws_p = pb.alloc_workspace(pb.pard_update_priority_workspace_bytes(len(s.pipes)), DEV)
    s.seed = seed
    return s


# ---- one pass -------------------------------------------------------------------------------------
def run(s):
    case = s.case
    if case["kind"] == "state":
        return run_state(s)
    if case["kind"] == "replay":
        return run_replay(s)
    if case["kind"] == "host":
        pb.pard_plan_host(s.pipes, s.req, s.n, s.state, s.n_ctx, 0, s.out, s.ws, stream=s.stream)
        return vars(s.out)
    if case["rule"]:
        pb.pard_plan_policy(s.pipes, s.req, s.arrivals, s.n, s.state, s.n_ctx, s.mode, s.out, s.ws, stream=s.stream)
    else:
        pb.pard_plan(s.pipes, s.req, s.n, s.state, s.n_ctx, s.mode, s.out, s.ws, stream=s.stream)
    pb.pard_goodput(None, s.out.seg_offsets, s.out.seg_kept, s.n, s.n_ctx, s.S, s.total, s.kept, stream=s.stream)
    return dict(vars(s.out), total=s.total, kept=s.kept)


def run_state(s):
    """The three refreshes of a State Planner's tick, enqueued one after the other."""
    case, st, nowait = s.case, s.state, pb.PARD_MODE_NOWAIT
    pb.pard_update_queue_delay(s.n_ctx, s.S, st.now_us, s.delay_time, s.delay, case["delay_samples"], WINDOW_US, nowait, s.q,
                               s.ws_q, stream=s.stream)
    pb.pard_update_priority(s.pipes, st.pipeline_of_ctx, s.n_ctx, s.S, st.batch, st.workers, s.history, case["history"],
                            min(5, case["history"]), 100_000, nowait, s.priority, s.ws_p, stream=s.stream)
    pb.pard_estimate_w(s.pipes, st.pipeline_of_ctx, s.n_ctx, s.S, s.R, s.waits, case["wait_samples"], 1, 10, s.seed, nowait,
                       s.w, s.ws_w, stream=s.stream)
    return {"q": s.q, "priority": s.priority, "w": s.w}


def run_replay(s):
    """One replay from its first epoch: the carried state starts over."""
    r = s.replay
    r.state.free_at_us.copy_(s.free_at)
    r.sample_time.fill_(-1)
    r.epoch = 0
    for e in range(EPOCHS):
        r.step(s.now[e], s.req[e], s.n, s.total[e], s.kept[e])
    return {"total": s.total, "kept": s.kept, "free_at": r.state.free_at_us, "sample_time": r.sample_time, "q": r.state.q_us}


# ---- what a pass cannot do without ----------------------------------------------------------------
def work(case):
    app, n_ctx = case["app"], case["n_ctx"]
    S, R = APPS[app][0], max(len(s) for s in slots(app))
    queues = n_ctx * S
    row = queues * (4 + 8 + 8 + 4) + n_ctx * (8 * R + 8)          # batch, free_at, q, workers; w, now
    if case["kind"] == "state":
        M, of = case["wait_samples"], [slots(app)[c % pipelines_used(case)] for c in range(n_ctx)]
        there = sum(graphs(app)[c % pipelines_used(case)][0] for c in range(n_ctx))
        return {"bytes": there * (4 * M + 4 * case["history"] + 1) + queues * (12 * case["delay_samples"] + 8)
                + 8 * sum(len(s) for s in of), "flops": float(M * sum(sum(s) for s in of))}
    # 16 bytes per request in; keep flag, estimate and order out (the kept indices depend on the load)
    per = 16 + 1 + 8 + 4 + (16 if case.get("rule") == "clipper" else 0)
    if case["kind"] == "replay":
        return {"bytes": EPOCHS * (16 * case["n"] + row), "flops": 0.0}
    return {"bytes": per * case["n"] + row + queues * 8 + 16 * n_ctx, "flops": 0.0}


def tolerance(case):
    return "exact"                           # whole numbers throughout
