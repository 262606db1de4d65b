"""Passes and segments of the tensor-core kNN, on the host: whatever the sizes, a query's
lists fit the merge kernel and all lists together stay within a fixed size."""
import ctypes

import pytest

import paper_2206_11408_gb300 as fg


def plan(n, m, nq, K, sms=152):
    out = (ctypes.c_int64 * 4)()
    f = fg.lib().fg_knn_plan
    f.restype = None
    f.argtypes = [ctypes.c_int64, ctypes.c_int, ctypes.c_int64, ctypes.c_int, ctypes.c_int,
                  ctypes.c_void_p]
    f(n, m, nq, K, sms, out)
    return tuple(out)


@pytest.mark.parametrize("K", [1, 16, 17, 40])
@pytest.mark.parametrize("m", [1, 96, 128, 960, 1024])
@pytest.mark.parametrize("n", [1, 128, 129, 60_000, 1_000_000, 3_500_000, 26_000_000, 100_000_000, 2**31 - 1])
def test_every_size_has_a_merge_and_bounded_lists(n, m, K):
    for nq in (1, 100, 128, 129, 10_000, 16_385, 1_000_000, 10_000_000, 2**31 - 1):
        for sms in (1, 132, 152, 600):
            KP, nseg, chunk, most_keys = plan(n, m, nq, K, sms)
            assert KP == (32 if K <= 16 else 64)
            assert 1 <= nseg <= (n + 127) // 128 and nseg * KP <= most_keys
            assert 1 <= chunk <= nq
            assert nseg * KP * 8 * chunk <= 512 << 20 or chunk <= 128
            assert -(-chunk // 128) * nseg < 2**31


def test_usual_sizes_take_one_pass():
    for n, m, nq in ((1_000_000, 128, 10_000), (1_000_000, 960, 1_000), (300_000, 96, 100_000)):
        for K in (10, 40):
            assert plan(n, m, nq, K)[2] == nq
