"""Shared memory of the planner that is spread over all SMs: every array has its place, and what is asked for covers them all.
(Host arithmetic of the test build of the library; no GPU.)"""
import ctypes as C

import numpy as np
import pytest

from paper_2310_09443_b200 import build

# what the kernel indexes, in the order of the layout: bytes for so many tiles of 64 slots and runs of 32 periods a block
ROUND, EDGE, SORT, TOP, LIMBS = 512, 1024, 12, 8, 4


def regions(tiles, runs, blocks, sorted_bytes):
    return [tiles * 16, runs * 512, ROUND * 4 * LIMBS, ROUND * 8, ROUND * 4, ROUND * 4, ROUND * 4, EDGE * 4, SORT * sorted_bytes,
            tiles * 4, tiles * 8, blocks * TOP * 4, blocks * TOP * 4, blocks * TOP, tiles * 512, tiles * 8, tiles * 4]


@pytest.fixture(scope="module")
def lib():
    lib = C.CDLL(build.build(hooks=True))
    lib.g10_test_spread_layout.restype = C.c_int32
    lib.g10_test_spread_layout.argtypes = [C.c_int64, C.c_int64, C.c_int32, C.POINTER(C.c_int64)]
    return lib


def test_arrays_do_not_overlap_and_end_inside(lib):
    rng = np.random.default_rng(5)
    cases = [(1_000_000, 1_025_000, 148), (900_000, 1_077_000, 148), (994_561, 1_022_977, 148), (2_097_151, 200_000, 148), (1, 1, 148), (64, 32, 1)]
    cases += [(int(np.exp(rng.uniform(0, np.log(2_097_151)))), int(np.exp(rng.uniform(0, np.log(1_500_000)))), int(rng.integers(1, 257))) for _ in range(5000)]
    out = (C.c_int64 * 18)()
    for K, periods, G in cases:
        sorted_bytes = lib.g10_test_spread_layout(K, periods, G, out)
        tiles, runs = -(-(-(-K // 64)) // G), -(-(-(-periods // G)) // 32)
        size = regions(tiles, runs, G, sorted_bytes)
        assert out[0] == 0 and sorted_bytes >= 64 * 8 + 65 * (8 + 8 + 4) + 8
        for j in range(17):
            assert out[j] % 16 == 0 and out[j] + size[j] <= out[j + 1], (K, periods, G, j)
