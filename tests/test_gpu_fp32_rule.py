"""FP32 fitness on both sides of the line between the tensor-core first layer and the CUDA cores (an estimate of a tile's
time in both, above a million first-layer products a spark): wide output layers and second layers at fan-ins where either
is the faster, against the oracle with the bar of tests/test_gpu_fp32_tc.py; and a spark's fitness is the same however
many share the launch, so the line does not depend on their number."""
import numpy as np
import pytest

import oracle
import workloads as W
from test_gpu_fp32_tc import case, evaluate, pkg  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("widths, act, n, count", [
    ((1024, 64, 32), "relu", 200, 9),      # 32 classes: tensor cores
    ((48, 64, 32), "relu", 700, 9),        # CUDA cores
    ((1024, 43, 25), "tanh", 129, 5),      # h1 no multiple of four
    ((784, 64, 24), "tanh", 257, 5),
    ((600, 96, 32), "tanh", 130, 3),
    ((128, 128, 32), "relu", 130, 4),
    ((1024, 64, 33, 16), "tanh", 140, 3),  # three layers, units no multiple of eight
    ((32, 64, 33, 16), "tanh", 600, 3),
    ((1024, 30, 7, 3), "relu", 131, 11),
    ((16, 43, 24, 5), "relu", 1600, 3),
    ((3072, 8, 64, 32), "tanh", 100, 2),   # one spark a tile, 8 of its columns used
    ((16, 8, 64, 32), "tanh", 8300, 2),
])
def test_both_sides_of_the_line(pkg, widths, act, n, count):  # noqa: F811
    w, X, y = case(widths, act, n)
    xs = W.random_vectors(count, w.dim, -1.0, 1.0, seed=5)
    want = oracle.Problem.for_workload(w, X, y).fitness_many(xs)
    got = evaluate(pkg, w, xs, X, y)
    assert np.all(np.abs(got - want) <= 4e-6 * np.abs(want) + 1e-7), (got, want)
    assert np.array_equal(got, np.concatenate([evaluate(pkg, w, xs[i:i + 1], X, y) for i in range(count)]))
