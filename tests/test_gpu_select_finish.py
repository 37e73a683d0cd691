"""Who finishes the guiding sparks' fitness means where no elite re-score does: the selection (up to two steps of 8
fireworks x 32 guiding sparks x 8 sample tiles) or a launch of its own.  Either way a captured generation ends bitwise in
the state of kernel-by-kernel launches, which always take the launch of its own."""
import numpy as np
import pytest

import workloads as W
from test_gpu_launch_path import _make, pkg  # noqa: F401

pytestmark = pytest.mark.gpu

GENS = 5


@pytest.mark.parametrize("mu, lam, m, n, runs, precision, fused", [
    (5, 40, 4, 512, 1, "fp32", True),       # one step
    (16, 8, 4, 100, 2, "fp32", True),       # two: sixteen fireworks
    (3, 128, 64, 512, 1, "fp32", True),     # two: 64 guiding sparks
    (5, 40, 4, 2048, 1, "fp32", True),      # two: sixteen sample tiles
    (17, 8, 4, 100, 1, "fp32", False),      # three
    (8, 132, 66, 1024, 1, "fp32", False),   # three
    (1, 8, 2, 2049, 1, "fp32", False),      # three: seventeen tiles
    (20, 8, 4, 1100, 3, "fp32", False),     # six
    (5, 16, 4, 512, 1, "bf16", True),       # low precision without the elite re-score
    (17, 16, 4, 512, 1, "bf16", False),
])
def test_graph_replay_equals_kernel_by_kernel(pkg, mu, lam, m, n, runs, precision, fused):  # noqa: F811
    low = precision == "bf16"
    w = W.scaled(W.MLP_784_64_10 if low else W.MLP_8_16_3, n_samples=n, n_fireworks=mu, sparks_per_firework=lam,
                 guiding_per_firework=m, eval_budget=W.budget_for_generations(mu, lam, m, GENS))
    if low:
        w = W.scaled(w, widths=(64, 64, 10), dim=W.mlp_param_count((64, 64, 10)))
    states = []
    for timed in (True, False):
        with _make(pkg, w, 41, pkg.MGFWA_BF16 if low else pkg.MGFWA_FP32,
                   dict(n_runs=runs, elite_rescore=0) if low else dict(n_runs=runs)) as h:
            if timed:
                h.profile(True)   # kernel-by-kernel launches between events
            h.run()
            info = h.info()
            states.append(([h.best(b) for b in range(runs)], h.read(pkg.MGFWA_BUF_FW_F), h.read(pkg.MGFWA_BUF_FW_X),
                           info.generations, info.kernel_launches))
    (ba, fa, xa, ga, la), (bb, fb, xb, gb, lb) = states
    assert ga == gb == GENS
    assert la - lb == GENS * (2 if fused else 1)   # the explosion's finish is the rank's in every captured generation
    assert np.array_equal(fa, fb) and np.array_equal(xa, xb)
    for (x1, f1, e1), (x2, f2, e2) in zip(ba, bb):
        assert np.array_equal(x1, x2) and f1 == f2 and e1 == e2
