"""Generations whose explosion is drawn in chunks beside the pair kernel (60 of its waves or more, at most two sparks to
a tile) end bitwise in the state of kernel-by-kernel launches, which draw and evaluate all sparks at once.  The sizes
leave a last chunk that is not whole and, E4M3, a last tile of one spark."""
import numpy as np
import pytest

import workloads as W
from test_gpu_launch_path import _make, pkg  # noqa: F401

pytestmark = pytest.mark.gpu

GENS = 3


@pytest.mark.parametrize("widths, n, mu, lam, m, precision, kw", [
    ((64, 128, 10), 2300, 5, 104, 8, "bf16", {"n_runs": 2}),
    ((64, 128, 20), 4096, 7, 95, 5, "fp8", {}),
    ((64, 128, 10), 4000, 7, 96, 8, "fp8", {"n_runs": 2, "loser_out": 1}),
    ((72, 128, 64, 10), 2048, 6, 200, 8, "bf16", {"loser_out": 1}),
    ((64, 128, 5), 2304, 8, 508, 4, "bf16", {}),                      # eight chunks
    ((64, 128, 64, 10), 2000, 7, 200, 8, "fp8", {"refine_every": 2, "refine_steps": 2, "refine_lr": 0.1}),
])
def test_graph_replay_equals_kernel_by_kernel(pkg, widths, n, mu, lam, m, precision, kw):  # noqa: F811
    w = W.scaled(W.MLP_784_64_10, widths=widths, acts=(W.ACT_RELU,) * (len(widths) - 2), n_samples=n, n_fireworks=mu,
                 sparks_per_firework=lam, guiding_per_firework=m,
                 eval_budget=W.budget_for_generations(mu, lam, m, GENS + 4 * ("refine_every" in kw)))
    prec = pkg.MGFWA_FP8 if precision == "fp8" else pkg.MGFWA_BF16
    states = []
    for timed in (True, False):
        with _make(pkg, w, 51, prec, kw) as h:
            if timed:
                h.profile(True)   # kernel-by-kernel launches between events
            assert h.pair_tile()[0] in (1, 2)
            h.step(GENS)
            info = h.info()
            states.append(([h.best(b) for b in range(h.cfg.n_runs)], h.read(pkg.MGFWA_BUF_FW_F),
                           h.read(pkg.MGFWA_BUF_FW_X), h.read(pkg.MGFWA_BUF_BEST_F), info.generations,
                           info.kernel_launches))
    (ba, fa, xa, bfa, ga, la), (bb, fb, xb, bfb, gb, lb) = states
    assert ga == gb == GENS
    # two launches a generation fewer (the means' finishes), two more for each chunk after the first
    chunks = 2 - (la - lb) / (2 * GENS)
    assert chunks == int(chunks) and 2 <= chunks <= 8, (la, lb)
    assert np.array_equal(fa, fb) and np.array_equal(xa, xb) and np.array_equal(bfa, bfb)
    for (x1, f1, e1), (x2, f2, e2) in zip(ba, bb):
        assert np.array_equal(x1, x2) and f1 == f2 and e1 == e2
