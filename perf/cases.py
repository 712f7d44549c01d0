"""The work that a user of the planner has it do, as cases to be timed.

A framework's compiler holds the kernel trace of a training step and asks, in this order: which tensors live when and how much
memory that takes (`analysis`, and `host_analysis` where the instrumented program left the trace in host memory), which tensors to
move away and bring back (`plan`; `cyclic` for a step that repeats; `batch` for the sensitivity of the plan to profiled times and
bandwidths), when to start the prefetches and where to put the instructions (`schedule`), and what the workload looks like
(`characterise`).  Traces are of two kinds: training steps of the shapes in `traces.py` (about a hundred to a few thousand kernels:
one launch after another on a nearly idle GPU) and random DAGs with the distributions of `traces.config4_stress_dag` (up to a
million kernels), drawn here on the GPU because they are made anew for every seed.

Every output is an integer and has to be the same bit for bit.
"""
import functools
import math

import numpy as np
import torch

from paper_2310_09443_b200 import binding as g10
from paper_2310_09443_b200 import traces

DEV = "cuda:0"


def listed():
    return [
        # the first two questions about a convolutional network's training step: a handful of launches on 1652 kernels
        dict(name="analysis_resnet", do="analysis", model="resnet", size=256),
        # a long trace of no round size with a few per cent of weights (many steps of a large model back to back)
        dict(name="analysis_dag_odd", do="analysis", model="dag", kernels=123457, tensors=370001, global_pct=3),
        # the largest: the stress trace of the benchmark
        dict(name="analysis_dag_1m", do="analysis", model="dag", kernels=1000000, tensors=4000000, global_pct=0),
        # the trace as the instrumented program wrote it, in pinned host memory; results wanted there too
        dict(name="host_analysis_vit", do="host_analysis", model="vit", size=4),
        # the workload figures (working set, idle periods by length and size) of a long trace
        dict(name="characterise_dag", do="characterise", model="dag", kernels=300000, tensors=1100000, global_pct=2),
        # eviction plans: the smallest step, a convolutional network, four transformer steps in a row, the stress trace
        dict(name="plan_mlp", do="plan", model="mlp", size=32, capacity_pct=40, host_gib=0),
        dict(name="plan_resnet", do="plan", model="resnet", size=256, capacity_pct=0, host_gib=0),
        dict(name="plan_vit", do="plan", model="vit", size=4, capacity_pct=0, host_gib=0),
        dict(name="plan_dag_1m", do="plan", model="dag", kernels=1000000, tensors=4000000, global_pct=0, capacity_pct=30, host_gib=0),
        # how far the plan depends on profiled times and on the links: one transformer step planned under many variants
        dict(name="batch_bert", do="batch", model="bert", size=24, capacity_pct=0, variants=96, jitter_pct=10),
        # the plan of a step that repeats (weights and optimizer state idle across the step's end)
        dict(name="cyclic_bert", do="cyclic", model="bert", size=24, capacity_pct=0, host_gib=0),
        # behind the plan: eager prefetches, then the instruction stream
        dict(name="schedule_dag", do="schedule", model="dag", kernels=200000, tensors=800000, capacity_pct=30, migrations=2000),
    ]


def _spread(rng, lo, hi):
    """A whole number between lo and hi, spread over the logarithm."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_step(rng, mlp_most=1000, vit_most=4):
    model = rng.choice(("mlp", "resnet", "bert", "vit") if vit_most else ("mlp", "resnet", "bert"))
    lo, hi = {"mlp": (8, mlp_most), "resnet": (16, 512), "bert": (2, 24), "vit": (1, max(vit_most, 1))}[model]
    return dict(model=model, size=_spread(rng, lo, hi))


def _draw_dag(rng, kernels_most, ratio_most=4.0):
    k = _spread(rng, 2000, kernels_most)
    return dict(model="dag", kernels=k, tensors=int(k * rng.uniform(1.2, ratio_most)))


def draw(rng):
    do = rng.choice(("analysis", "analysis", "host_analysis", "characterise", "plan", "plan", "plan", "batch", "cyclic", "schedule"))
    if do in ("analysis", "host_analysis", "characterise"):
        if rng.random() < 0.4:
            return dict(do=do, **_draw_step(rng))
        most = {"analysis": 1000000, "host_analysis": 200000, "characterise": 500000}[do]
        return dict(do=do, global_pct=rng.choice((0, 1, 5)), **_draw_dag(rng, most))
    pct = rng.randrange(25, 66)
    if do == "plan":
        if rng.random() < 0.65:
            return dict(do=do, capacity_pct=pct, host_gib=rng.choice((0, 0, 8)), **_draw_step(rng))
        return dict(do=do, capacity_pct=pct, host_gib=0, global_pct=rng.choice((0, 1)), **_draw_dag(rng, 200000))
    if do == "batch":
        return dict(do=do, capacity_pct=pct, variants=_spread(rng, 8, 148), jitter_pct=rng.choice((5, 10, 25)), **_draw_step(rng, 256, 0))
    if do == "cyclic":
        return dict(do=do, capacity_pct=pct, host_gib=rng.choice((0, 0, 8)), **_draw_step(rng, 500, 1))
    dag = _draw_dag(rng, 250000)
    dag["tensors"] = max(dag["tensors"], 3 * dag["kernels"])
    return dict(do="schedule", capacity_pct=30, migrations=int(20 * dag["kernels"] ** 0.36), **dag)


# ---- traces ----------------------------------------------------------------------------------------------------------
def _step(case, seed):
    """A training step of one of the shapes that the repository names, `size` being layers, batch or steps in a row."""
    model, size = case["model"], case["size"]
    if model == "mlp":
        return traces.config0_mlp_chain(seed, layers=size)
    if model == "resnet":
        return traces.config1_resnet152(seed, batch=size)
    if model == "bert":
        if size == 24:
            return traces.config2_bert_large(seed)
        return traces._transformer("c2_bert_%d" % size, seed, size, 128, 512, 1024, 16, 4096, 2, 24 * traces.GiB, 1)
    return traces.config3_vit_huge(seed, iterations=size)


def _dag(case, seed):
    """The random DAG of traces.config4_stress_dag, drawn on the GPU, with `global_pct` per cent of weights among its tensors."""
    K, N, pct = case["kernels"], case["tensors"], case.get("global_pct", 0)
    gen = torch.Generator(device=DEV)
    gen.manual_seed(seed)
    uniform = lambda n: torch.rand(n, generator=gen, device=DEV, dtype=torch.float64)
    normal = lambda n: torch.randn(n, generator=gen, device=DEV, dtype=torch.float64)
    geometric = lambda n, p: torch.floor(torch.log1p(-uniform(n)) / math.log1p(-p)).long() + 1
    birth = torch.cat([torch.arange(K, device=DEV), torch.randint(0, K, (N - K,), generator=gen, device=DEV)])
    long_lived = uniform(N) < 0.05
    reuse = geometric(N, 0.8) - 1
    alive, cur = torch.arange(N, device=DEV), birth
    ev = [cur * N + alive]
    lo, hi = max(1, K // 100), max(2, K // 2)
    j = 0
    while True:
        keep = reuse[alive] > j
        alive, cur = alive[keep], cur[keep]
        if not alive.numel():
            break
        gap = torch.where(long_lived[alive], torch.randint(lo, hi + 1, (alive.numel(),), generator=gen, device=DEV),
                          geometric(alive.numel(), 1.0 / 64.0))
        cur = cur + gap
        keep = cur < K
        alive, cur = alive[keep], cur[keep]
        ev.append(cur * N + alive)
        j += 1
    key = torch.sort(torch.cat(ev)).values
    ptr = torch.searchsorted(key, torch.arange(K + 1, device=DEV) * N)
    size = torch.floor(torch.exp(math.log(4 << 20) + 1.5 * normal(N))).clamp(4096, 2 << 30).long()
    ns = torch.floor(torch.exp(math.log(100_000.0) + normal(K))).clamp(min=1).long()
    glob = (uniform(N) < pct / 100.0).to(torch.uint8)
    return g10.TraceBuffers(ptr, (key % N).int(), size, ns, glob)


def _room(case, tb):
    """(events, migrations) that a program which analyses one trace after another keeps buffers for: the DAG's events differ in
    number from seed to seed, those of a training step do not."""
    return (tb.E, tb.E) if case["model"] != "dag" else (int(1.3 * tb.N) + 1000, tb.K // 2)


def _trace(case, seed):
    """(trace on the GPU, host and SSD bandwidth, the capacity that the configuration names or None)"""
    if case["model"] == "dag":
        return _dag(case, seed), traces.HOST_BW, traces.SSD_BW, None
    t = _step(case, seed)
    return g10.upload(t, DEV), t.host_bw, t.ssd_bw, t.capacity_bytes


def _pinned(tb):
    pin = lambda t: t.cpu().pin_memory()
    return g10.TraceBuffers(pin(tb.kernel_ptr), pin(tb.kernel_tensors), pin(tb.tensor_bytes), pin(tb.kernel_ns), pin(tb.tensor_global))


def _capacity(case, tb, named):
    if not case["capacity_pct"]:
        return named
    return int(g10.g10_pressure_timeline(tb).peak_bytes.item()) * case["capacity_pct"] // 100


def _workspace(which, tb):
    return torch.empty(max(256, g10.g10_workspace_bytes(which, tb.K, tb.N, tb.E, tb.mem)), dtype=torch.uint8, device=DEV)


def _cleared(r):
    """The result buffers of an earlier call, emptied: a program that analyses trace after trace keeps them."""
    for t in vars(r).values():
        if isinstance(t, torch.Tensor):
            t.zero_()
        elif hasattr(t, "__dict__"):
            _cleared(t)
    return r


# ---- a user's program ------------------------------------------------------------------------------------------------
def prepare(case, seed):
    do = case["do"]
    tb, host_bw, ssd_bw, named = _trace(case, seed)
    s = dict(do=do, tb=tb, bw=(host_bw, ssd_bw))
    if do in ("analysis", "host_analysis"):
        if do == "host_analysis":
            tb = s["tb"] = _pinned(tb)
        s["ws"] = _workspace(g10.WS_ANALYSIS, tb)
        s["room"] = _room(case, tb)[0]
        s["out"] = _cleared(g10.g10_vitality(tb, ws=s["ws"], timeline=True, device=DEV, uses_cap=s["room"], periods_cap=s["room"]))
        s["timeline"] = s["out"].timeline
        return s
    if do == "characterise":
        v = g10.g10_vitality(tb, timeline=True)
        uses, periods = (int(x) for x in v.counts[:2].tolist())
        s["args"] = (tb.K, tb.N, v.use_ptr, v.uses[:uses], tb.tensor_bytes, v.timeline.kernel_start_ns, periods,
                     v.period_tensor[:periods], v.period_prev_use[:periods], v.period_next_use[:periods], host_bw, ssd_bw)
        return s
    s["capacity"] = _capacity(case, tb, named)
    s["host"] = case.get("host_gib", 0) << 30
    if do == "batch":
        rng = np.random.default_rng(seed)
        ns = tb.kernel_ns.double()
        s["variants"] = [dict(gpu_capacity_bytes=s["capacity"], host_bw=host_bw, ssd_bw=ssd_bw)]
        for _ in range(case["variants"] - 1):
            f = torch.from_numpy(1.0 + (2.0 * rng.random(tb.K) - 1.0) * case["jitter_pct"] / 100.0).to(DEV)
            s["variants"].append(dict(gpu_capacity_bytes=s["capacity"], host_bw=host_bw, ssd_bw=int(rng.choice((ssd_bw, 2 * ssd_bw))),
                                      kernel_ns=torch.round(ns * f).clamp(min=1).long()))
        s["ws"] = _workspace(g10.WS_BATCH, tb)
        s["plans"] = np.zeros((case["variants"], tb.E // 2, 48), dtype=np.uint8)
        return s
    s["ws"] = _workspace(g10.WS_PLAN, tb)
    if do == "cyclic":
        s["plans"] = np.zeros((tb.E, 48), dtype=np.uint8)
        return s
    if do == "plan":
        s["room"] = _room(case, tb)[1]
        s["out"] = _cleared(g10.g10_plan_migrations(tb, s["capacity"], host_bw, ssd_bw, ws=s["ws"], max_iterations=1, migrations_cap=s["room"]))
        return s
    v = g10.g10_vitality(tb, timeline=True)
    # (so many migrations and no more, for every seed the same number: most of the plan in the listed case)
    plan = g10.g10_plan_migrations(tb, s["capacity"], host_bw, ssd_bw, ws=s["ws"], max_iterations=case["migrations"])
    n = int(plan.summary[0].item())
    s.update(v=v, plan=plan, migrations=n)
    s["ws_prefetch"] = torch.empty(max(256, g10.g10_workspace_bytes(g10.WS_PREFETCH, tb.K, 0, n)), dtype=torch.uint8, device=DEV)
    s["ws_emit"] = torch.empty(max(256, g10.g10_workspace_bytes(g10.WS_EMIT, tb.K, tb.N, n)), dtype=torch.uint8, device=DEV)
    return s


def _analysis(v, t):
    return dict(first=v.first_use, last=v.last_use, num=v.num_uses, use_ptr=v.use_ptr, uses=v.uses, period_ptr=v.period_ptr,
                period_tensor=v.period_tensor, prev=v.period_prev_use, next=v.period_next_use, counts=v.counts, start=t.kernel_start_ns,
                pressure=t.pressure, peak=t.peak_bytes, slot=t.peak_slot, status=t.status)


def _keep(table, records):
    table[: records.shape[0]] = records.view(np.uint8).reshape(-1, 48)


def run(s):
    do, tb, (host_bw, ssd_bw) = s["do"], s["tb"], s["bw"]
    if do in ("analysis", "host_analysis"):
        v = g10.g10_vitality(tb, ws=s["ws"], out=s["out"], timeline=s["timeline"], device=DEV, uses_cap=s["room"], periods_cap=s["room"])
        return _analysis(v, s["timeline"])
    if do == "characterise":
        r = g10.g10_characterize(*s["args"])
        return dict(active=r.active_bytes, lengths=r.len_hist, sizes=r.size_len_hist, hide=r.hide, summary=r.summary)
    if do == "plan":
        r = g10.g10_plan_migrations(tb, s["capacity"], host_bw, ssd_bw, host_capacity_bytes=s["host"], ws=s["ws"], out=s["out"],
                                    migrations_cap=s["room"])
        return dict(migrations=r.migrations, pressure=r.final_pressure, summary=r.summary)
    if do == "cyclic":
        r = g10.g10_plan_cyclic(tb, s["capacity"], host_bw, ssd_bw, host_capacity_bytes=s["host"], ws=s["ws"])
        # the compiler reads the plan
        _keep(s["plans"], g10.migrations_numpy(r))
        return dict(migrations=s["plans"], pressure=r.final_pressure, summary=r.summary)
    if do == "batch":
        r = g10.g10_plan_batch(tb, s["variants"], ws=s["ws"])
        # the study reads every variant's plan
        for v in range(len(s["variants"])):
            _keep(s["plans"][v], g10.batch_migrations_numpy(r, v))
        return dict(migrations=s["plans"], pressure=r.final_pressure, summary=r.summary, stability=r.stability)
    v, plan, n = s["v"], s["plan"], s["migrations"]
    # (the pass changes the pressure curve that it is given: a fresh copy for each pass)
    p = g10.g10_schedule_prefetch(tb.K, n, plan.migrations, v.timeline.kernel_start_ns, tb.tensor_bytes, s["capacity"],
                                  plan.final_pressure.clone(), ws=s["ws_prefetch"])
    e = g10.g10_emit_instructions(tb.K, tb.N, v.first_use, v.last_use, tb.tensor_bytes, tb.tensor_global, v.timeline.kernel_start_ns,
                                  n, plan.migrations, p.new_prefetch_issue_ns, ws=s["ws_emit"])
    # (every tensor of these traces is used and none is a weight: all records of the buffer are written)
    return dict(pressure=p.pressure, order=p.order, last=p.new_absent_last, issue=p.new_prefetch_issue_ns, moved=p.summary,
                inst_ptr=e.inst_ptr, instructions=e.instructions, counts=e.counts)


# ---- what a pass cannot do without -----------------------------------------------------------------------------------
@functools.lru_cache(maxsize=None)
def _step_sizes(model, size):
    t = _step(dict(model=model, size=size), 0)
    return t.K, t.N, t.E


def work(case):
    """Bytes of the inputs read once and the outputs written once; every operation is an integer one.  What only the data decides is
    taken at its mean: uses and periods of the DAG's tensors (0.25 reuses each), a migration for every second kernel of a training
    step and for every 75th of a DAG."""
    if case["model"] == "dag":
        K, N = case["kernels"], case["tensors"]
        E, periods, moves = int(1.246 * N), int(0.242 * N), case.get("migrations", K // 75)
    else:
        K, N, E = _step_sizes(case["model"], case["size"])
        periods, moves = E // 2, K // 2
    trace = 8 * (K + 1) + 4 * E + 9 * N + 8 * K
    analysis = 12 * N + 16 * (N + 1) + 4 * E + 12 * periods + 24 + 8 * (K + 1) + 8 * K + 20
    plan = 48 * moves + 8 * K + 64
    do = case["do"]
    if do in ("analysis", "host_analysis"):
        n = trace + analysis
    elif do == "characterise":
        n = 8 * (N + 1) + 4 * E + 8 * N + 8 * (K + 1) + 12 * periods + 8 * K
    elif do in ("plan", "cyclic"):
        n = trace + plan
    elif do == "batch":
        n = trace + case["variants"] * (8 * K + plan + 16)
    else:
        n = 8 * K + 56 * moves + 8 * K + 16 * moves + (8 * (K + 1) + 17 * N + 56 * moves) + 8 * (K + 2) + 32 * 2 * (N + moves)
    return {"bytes": n, "flops": 0}


def tolerance(case):
    return "exact"
