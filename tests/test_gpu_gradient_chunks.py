"""Weight gradients on both sides of the line between 64- and 128-sample chunks (output tiles times 128-sample chunks
against two thirds of the SMs: 101.3 blocks on 152), against the oracle's FP64 backpropagation with the bar of
tests/test_gpu_refine.py."""
import numpy as np
import pytest

import oracle
import workloads as W
from test_gpu_refine import _net, pkg  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("widths, N, R", [
    ((16, 64, 3), 129, 2),           # one tile: 64-sample chunks, the last of one sample
    ((120, 64, 10), 2048, 2),        # one tile, 32 chunks of 64
    ((640, 64, 10), 2048, 1),        # six tiles, 96 blocks: 64
    ((768, 64, 10), 1920, 3),        # seven tiles (769 rows), 105 blocks: 128
    ((784, 64, 10), 2048, 1),        # seven tiles, 112 blocks: 128
    ((120, 128, 24, 5), 511, 2),     # three layers: one and two tiles, a ragged chunk
])
def test_gradient_on_both_sides_of_the_line(pkg, widths, N, R):  # noqa: F811
    w = _net(widths, (W.ACT_TANH,) * (len(widths) - 2), N)
    X, y = W.make_data(w)
    prob = oracle.Problem.for_workload(w, X, y)
    xs = W.random_vectors(R, w.dim, -0.5, 0.5, 7)
    with pkg.Mgfwa.for_workload(w, 1, X=X, y=y, n_runs=R, refine_every=1, refine_steps=1, refine_lr=0.1) as h:
        f, g = h.gradient(xs)
    for r in range(R):
        fo, go = oracle.gradient(prob, xs[r])
        mx = np.max(np.abs(go))
        assert abs(f[r] - fo) <= 1e-5 * abs(fo) + 1e-5
        assert np.all(np.abs(g[r] - go) <= 1e-5 * mx + 1e-4 * np.abs(go)), (r, np.max(np.abs(g[r] - go)) / mx)
