"""FP32 fitness on the tensor cores where the first layer's sums are whole numbers of up to 20 bits (times a power of
two): nothing may be lost or added.  Batches of one 128-sample tile stay below the tensor-core kernel's line, so the CUDA-core kernel gives each
tile's loss sum (a mean over 128 is an exact division); from there on both kernels compute with the same operations in
the same order, so the whole batch's fitness is bitwise the tiles' sums added in order."""
import numpy as np
import pytest

import workloads as W
from test_gpu_fp32_tc import case, evaluate, pkg  # noqa: F401

pytestmark = pytest.mark.gpu


# nonzeros * x_max * w_max < 2^20, so that every sum on the way is such a number too
@pytest.mark.parametrize("widths, act, nonzeros, x_max, w_max", [
    ((64, 64, 10), "relu", 64, 1, 8),            # binary inputs, weights in eighths
    ((64, 64, 10), "tanh", 64, 255, 63),         # one BF16 part each
    ((64, 40, 24, 3), "relu", 64, 2047, 7),      # inputs of two parts
    ((64, 17, 32), "relu", 64, 3, 5461),         # weights of two parts
    ((64, 64, 5), "relu", 4, 1, (1 << 18) - 1),  # weights of three parts
    ((248, 32, 4), "relu", 1, 1, (1 << 20) - 1),  # one-hot inputs
])
def test_exact_sums_stay_exact(pkg, widths, act, nonzeros, x_max, w_max):  # noqa: F811
    n = 128 * -(-(1 << 20) // (widths[0] * widths[1] * 128))   # the least whole number of tiles on the line
    assert n >= 256
    w, X, y = case(widths, act, n)
    rng = np.random.default_rng(x_max)
    X = np.zeros_like(X)
    for r in X:
        r[rng.choice(widths[0], nonzeros, replace=False)] = rng.integers(1, x_max + 1, nonzeros)
    xs = W.random_vectors(9, w.dim, -1.0, 1.0, seed=7)
    k = widths[0] * widths[1]
    scale = 2.0 ** -(int(nonzeros * x_max * w_max).bit_length() - 3)
    xs[:, :k] = (rng.integers(-w_max, w_max + 1, (9, k)) * scale).astype(np.float32)
    got = evaluate(pkg, w, xs, X, y)
    total = None
    for t in range(n // 128):
        s = slice(128 * t, 128 * (t + 1))
        one = W.scaled(w, n_samples=128)
        tile = evaluate(pkg, one, xs, np.ascontiguousarray(X[s]), np.ascontiguousarray(y[s])) * np.float32(128)
        total = tile if total is None else total + tile
    assert np.array_equal(got, total / np.float32(n))
