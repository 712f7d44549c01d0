"""Blocks of the planners' grids that fall behind.  Every block takes the same decisions from the same data: what one block changes
for the next iteration must not be seen by another that still decides this one.  A test build of the library
(-DG10_TEST_HOOKS, never loaded by the binding) lets one block come 50 us late to every choice, which is several
iterations' worth; the plan has to be the oracle's all the same.  Every wait is bounded as always."""
import ctypes as C

import numpy as np
import pytest

from paper_2310_09443_b200 import traces

pytestmark = pytest.mark.gpu

FLAG_GLOBAL_STATE, FLAG_SPREAD_STATE = 0x2, 0x8
FLAG_TEST_LATE_BLOCK = 0x20000000


def near_ties(groups=3, K=300, n=7000):
    """`groups` crowds of periods, one after the other; in each all periods have the same rounded score and the exact comparison
    decides (an odd byte makes the transfer time round up).  A commit takes the SSD, then the host, from all the others."""
    rng = np.random.default_rng(8)
    size = (1 << 33) + 16 * rng.integers(0, 1 << 18, size=groups * n) + (np.arange(groups * n) % 3 < 2)
    deg = np.zeros(groups * K, np.int64)
    for g in range(groups):
        deg[g * K + 2] = deg[g * K + K - 3] = n
    tensors = np.concatenate([np.tile(np.arange(g * n, (g + 1) * n, dtype=np.int32), 2) for g in range(groups)])
    return traces.Trace(name="ties", kernel_ptr=np.concatenate([[0], np.cumsum(deg)]), kernel_tensors=tensors, tensor_bytes=size.astype(np.int64),
                        kernel_ns=np.full(groups * K, 50_000_001, np.int64), tensor_global=np.zeros(groups * n, np.uint8),
                        host_bw=16_000_000_000, ssd_bw=3_200_000_000, capacity_frac=(1, 2))


@pytest.mark.parametrize("flags", [FLAG_SPREAD_STATE, FLAG_GLOBAL_STATE])
def test_a_late_block_decides_as_the_others(oracle, flags):
    import torch
    from paper_2310_09443_b200 import binding, build
    build.build()
    binding.load_library()
    hooks = C.CDLL(build.build(hooks=True))
    hooks.g10_plan_migrations.restype = C.c_int32
    hooks.g10_plan_migrations.argtypes = [C.POINTER(binding._Trace), C.c_uint64, C.c_uint64, C.c_uint64, C.POINTER(binding._Options),
                                          C.POINTER(binding._PlanOut), C.c_void_p, C.c_size_t, C.c_void_p]
    tr = near_ties()
    tb = binding.upload(tr)
    start, P0, peak, slot = oracle.timeline(tr)
    cap = tr.capacity_from_peak(peak)
    ref = oracle.plan(tr, cap, lazy=True)
    assert len(ref.migrations) == 6
    ws = torch.zeros(binding.g10_workspace_bytes(binding.WS_PLAN, tb.K, tb.N, tb.E), dtype=torch.uint8, device="cuda")
    mig = torch.zeros(tb.E * 48, dtype=torch.uint8, device="cuda")
    finalp = torch.zeros(tb.K, dtype=torch.int64, device="cuda")
    summary = torch.zeros(8, dtype=torch.int64, device="cuda")
    po = binding._PlanOut(mig.data_ptr(), tb.E, finalp.data_ptr(), summary.data_ptr())
    for late in (0, FLAG_TEST_LATE_BLOCK, FLAG_TEST_LATE_BLOCK):
        opt = binding._Options(0, 0, flags | late, None, 0)
        assert hooks.g10_plan_migrations(C.byref(tb.c_struct()), cap, tr.host_bw, tr.ssd_bw, C.byref(opt), C.byref(po), ws.data_ptr(), ws.numel(),
                                         torch.cuda.current_stream().cuda_stream) == 0
        torch.cuda.synchronize()
        s = summary.cpu().numpy()
        assert s[7] == 0 and np.array_equal(s[:7], ref.summary[:7])
        assert np.array_equal(mig[:int(s[0]) * 48].cpu().numpy().view(binding.MIGRATION_DTYPE), ref.migrations)
        assert np.array_equal(finalp.cpu().numpy(), ref.final_pressure)
