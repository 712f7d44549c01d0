"""Calls after cudaDeviceReset.  A reset takes back what kernels were allowed (shared memory, cluster sizes): the library has to
allow it again, not remember that it did.  In a process of its own, with a test build of the library (-DG10_TEST_HOOKS) whose
own runtime does the reset and holds the device memory."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = """
import ctypes as C
import numpy as np
from paper_2310_09443_b200 import binding, build, traces
from oracle import g10_oracle as oracle
oracle.build()
binding.LIB_PATH = build.build(hooks=True)
lib = binding.load_library()
lib.g10_test_upload.restype = C.c_void_p
lib.g10_test_upload.argtypes = [C.c_void_p, C.c_size_t]
lib.g10_test_download.argtypes = [C.c_void_p, C.c_void_p, C.c_size_t]
tr = traces.config0_mlp_chain()
start, P0, peak, slot = oracle.timeline(tr)
cap = tr.capacity_from_peak(peak)
ov = oracle.vitality(tr.kernel_ptr, tr.kernel_tensors, tr.N)
ct = binding._Trace(tr.K, tr.N, tr.E, tr.kernel_ptr.ctypes.data, tr.kernel_tensors.ctypes.data, tr.tensor_bytes.ctypes.data,
                    tr.kernel_ns.ctypes.data, tr.tensor_global.ctypes.data, binding.MEM_HOST)


def plans():
    n = binding.g10_workspace_bytes(binding.WS_PLAN, tr.K, tr.N, tr.E, binding.MEM_HOST)
    ws = lib.g10_test_upload(None, n)
    for call, flags, ref in ((lib.g10_plan_migrations, 0, oracle.plan(tr, cap)), (lib.g10_plan_migrations, binding.FLAG_MULTI_BLOCK, oracle.plan(tr, cap)),
                             (lib.g10_plan_migrations, binding.FLAG_SPREAD_STATE, oracle.plan(tr, cap)),
                             (lib.g10_plan_migrations, binding.FLAG_GLOBAL_STATE, oracle.plan(tr, cap)), (lib.g10_plan_cyclic, 0, oracle.plan_cyclic(tr, cap))):
        mig, P, s = np.zeros(tr.E, binding.MIGRATION_DTYPE), np.zeros(tr.K, np.int64), np.zeros(8, np.int64)
        po = binding._PlanOut(mig.ctypes.data, tr.E, P.ctypes.data, s.ctypes.data)
        opt = binding._Options(0, 0, flags, None, 0)
        rc = call(C.byref(ct), cap, tr.host_bw, tr.ssd_bw, C.byref(opt), C.byref(po), ws, n, None)
        assert rc == 0, (flags, rc)
        assert s[7] == 0 and np.array_equal(s[:7], ref.summary[:7]) and np.array_equal(mig[:s[0]], ref.migrations) and np.array_equal(P, ref.final_pressure)


def statistics():
    up = lambda a: lib.g10_test_upload(np.ascontiguousarray(a).ctypes.data, max(a.nbytes, 8))
    sizes = [tr.K, 64, 41 * 45, 2, 2]
    outs = [lib.g10_test_upload(None, 8 * n) for n in sizes]
    so = binding._StatsOut(*outs)
    rc = lib.g10_characterize(tr.K, tr.N, up(ov.use_ptr), up(ov.uses), up(tr.tensor_bytes), up(start), len(ov.period_tensor), up(ov.period_tensor),
                              up(ov.period_prev_use), up(ov.period_next_use), tr.host_bw, tr.ssd_bw, C.byref(so), None)
    assert rc == 0, rc
    got = [np.zeros(n, np.int64) for n in sizes]
    for a, p in zip(got, outs):
        assert lib.g10_test_download(a.ctypes.data, p, a.nbytes) == 0
    oc = oracle.characterize(tr.K, ov, tr.tensor_bytes, start, tr.host_bw, tr.ssd_bw)
    for a, b in zip(got, (oc.active_bytes, oc.len_hist, oc.size_len_hist, oc.hide, oc.summary)):
        assert np.array_equal(a, np.asarray(b).ravel())


for _ in range(3):
    plans()
    statistics()
    assert lib.g10_test_device_reset() == 0
print("fine")
"""


def test_calls_after_a_device_reset():
    r = subprocess.run([sys.executable, "-c", CHILD], cwd=ROOT, env=dict(os.environ, PYTHONPATH=ROOT), capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "fine" in r.stdout, r.stdout + r.stderr
