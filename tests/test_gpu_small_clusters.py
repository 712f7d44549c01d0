"""Devices that cannot place a cluster of 16 blocks (a part of a GPU may not): the planner of one cluster takes the largest that
they can, and the planners behind it do the work where the trace does not fit that, or where there is none at all.  A test
build of the library (-DG10_TEST_HOOKS) takes an environment variable for the device's answer."""
import os

import numpy as np
import pytest

import test_gpu_parity as P
from paper_2310_09443_b200 import traces

pytestmark = pytest.mark.gpu


@pytest.fixture(params=[0, 1, 4])
def gpu(request, monkeypatch):
    from paper_2310_09443_b200 import binding, build
    monkeypatch.setattr(binding, "LIB_PATH", build.build(hooks=True))
    monkeypatch.setattr(binding, "_lib", None)
    monkeypatch.setenv("G10_TEST_MAX_CLUSTER", str(request.param))
    binding.load_library()
    binding.most_blocks = request.param
    yield binding
    del binding.most_blocks


def test_smaller_clusters_or_none(gpu, oracle):
    tr = traces.config1_resnet152()
    start, P0, peak, slot = oracle.timeline(tr)
    cap = tr.capacity_from_peak(peak)
    tb = gpu.upload(tr)
    ref = oracle.plan(tr, cap, lazy=True)
    for flags in (0, gpu.FLAG_MULTI_BLOCK):
        P.check_plan(gpu, tr, tb, cap, ref, flags=flags)
    before = gpu.g10_launch_count()
    gpu.g10_plan_migrations(tb, cap, tr.host_bw, tr.ssd_bw)
    # (one launch for the analysis and one for the plan where the host knows that the trace fits the cluster)
    assert (gpu.g10_launch_count() - before == 2) == (gpu.most_blocks == 4)
    base = dict(gpu_capacity_bytes=cap, host_bw=tr.host_bw, ssd_bw=tr.ssd_bw)
    P.check_batch(gpu, oracle, tr, [base, dict(base, ssd_bw=2 * tr.ssd_bw)], max_iterations=60)
    P.check_stats(gpu, oracle, tr)
    tr = traces.config0_mlp_chain()
    start, P0, peak, slot = oracle.timeline(tr)
    P.check_cyclic(gpu, oracle, tr, tr.capacity_from_peak(peak))
    P.check_stats(gpu, oracle, traces.random_toy(np.random.default_rng(3), 20000, 300, max_deg=3))
    assert os.environ["G10_TEST_MAX_CLUSTER"] == str(gpu.most_blocks)
