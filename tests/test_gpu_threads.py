"""Threads of one process, each with a stream, traces and buffers of its own, in the same call at the same time: traces of
different sizes ask for different amounts of shared memory of the same kernels, and what one thread allows a kernel must not take
away what another has just been allowed."""
import threading

import numpy as np
import pytest

from paper_2310_09443_b200 import traces

pytestmark = pytest.mark.gpu

REPEATS = 2000


@pytest.fixture(scope="module")
def gpu():
    from paper_2310_09443_b200 import binding, build
    build.build()
    binding.load_library()
    return binding


def _trace(K, N, seed):
    """Every tensor used at two to four kernels."""
    rng = np.random.default_rng(seed)
    lists = [[] for _ in range(K)]
    for i in range(N):
        for k in sorted(set(int(x) for x in rng.integers(0, K, size=int(rng.integers(2, 5))))):
            lists[k].append(i)
    return traces.from_lists("threads", lists, rng.integers(1 << 16, 1 << 24, size=N), rng.integers(10_000, 3_000_000, size=K),
                             np.zeros(N, np.uint8), capacity_frac=(2, 5))


def _results(r, names):
    return [getattr(r, n) for n in names]


def _prepared(gpu, oracle, call, K, N):
    """A function of no arguments that makes the call once; returns tensors that are the same every time."""
    tr = _trace(K, N, K + N)
    tb = gpu.upload(tr)
    start, P0, peak, slot = oracle.timeline(tr)
    cap = tr.capacity_from_peak(peak)
    if call == "vitality":
        return lambda: _results(gpu.g10_vitality(tb), ("first_use", "last_use", "num_uses", "use_ptr", "period_ptr", "counts"))
    if call == "batch":
        variants = [dict(gpu_capacity_bytes=cap, host_bw=tr.host_bw, ssd_bw=tr.ssd_bw)] * 2
        return lambda: _results(gpu.g10_plan_batch(tb, variants, max_iterations=3), ("summary", "stability", "final_pressure"))
    v = gpu.g10_vitality(tb, timeline=True)
    plan = gpu.g10_plan_migrations(tb, cap, tr.host_bw, tr.ssd_bw, max_iterations=40)
    n = int(plan.summary[0].item())
    if call == "emit":
        return lambda: _results(gpu.g10_emit_instructions(tr.K, tr.N, v.first_use, v.last_use, tb.tensor_bytes, tb.tensor_global,
                                                          v.timeline.kernel_start_ns, n, plan.migrations), ("inst_ptr", "counts"))
    return lambda: _results(gpu.g10_schedule_prefetch(tr.K, n, plan.migrations, v.timeline.kernel_start_ns, tb.tensor_bytes, cap,
                                                      plan.final_pressure.clone(), one_block=call == "prefetch_one_block"),
                            ("pressure", "order", "new_absent_last", "new_prefetch_issue_ns", "summary"))


@pytest.mark.parametrize("call,sizes", [("vitality", ((9000, 30_000), (40_000, 400_000))), ("emit", ((300, 2000), (5000, 40_000))),
                                        ("prefetch", ((300, 2000), (5000, 12_000))), ("prefetch_one_block", ((300, 2000), (5000, 12_000))),
                                        ("batch", ((64, 300), (300, 2000)))])
def test_threads_with_different_sizes(gpu, oracle, call, sizes):
    import torch
    once = [_prepared(gpu, oracle, call, *s) for s in sizes]
    torch.cuda.synchronize()
    want = [[t.clone() for t in f()] for f in once]
    torch.cuda.synchronize()
    failed = []
    once, want = [once[0], once[0], once[1]], [want[0], want[0], want[1]]          # two small ones for every large one
    begin = threading.Barrier(len(once))

    def work(f, ref):
        try:
            s = torch.cuda.Stream()
            with torch.cuda.stream(s):
                begin.wait()
                for _ in range(REPEATS):
                    got = f()
                for a, b in zip(got, ref):
                    assert torch.equal(a, b)
            s.synchronize()
        except Exception as e:
            failed.append(repr(e))

    threads = [threading.Thread(target=work, args=p) for p in zip(once, want)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed, failed
