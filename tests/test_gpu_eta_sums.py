"""Sums of eta = W^T [Q | r] in the mixed solves: the rows' products are FP32 pairs, and for blocks narrower than four
columns the sums over the threads are FP64, so that rows of 2^50, 2^26 and 1 (which no pair holds together) add exactly."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("k", [1, 2, 3, 5])
@pytest.mark.parametrize("n", [3, 61, 1000, 5000])
def test_thread_sums_are_fp64(n, k):
    import device_kernels
    rng = np.random.default_rng(n + k)
    w = rng.choice([2.0 ** 50, -(2.0 ** 50), 2.0 ** 26, 1.0], size=(n, k))
    w[: n // 2] = np.where(np.abs(w[: n // 2]) > 1.0, w[: n // 2], -1.0)
    # partial sums stay below 2^53, whatever the order: at most four rows of 2^50 a column
    for c in range(k):
        big = np.flatnonzero(np.abs(w[:, c]) == 2.0 ** 50)
        w[big[4:], c] = 1.0
    Q, r = np.ones((n, k)), np.ones(n)
    d = [torch.from_numpy(x).cuda() for x in (w, Q, r)]
    out = np.zeros((k, k + 1))
    lib = device_kernels.load()
    rc = lib.t_eta(n, k, *(ctypes.c_void_p(x.data_ptr()) for x in d), 1, out.ctypes.data_as(ctypes.c_void_p))
    assert rc == 0
    assert np.array_equal(out, np.repeat(w.sum(axis=0)[:, None], k + 1, axis=1))
