"""FP32X3 layers at every way their K splits meet: one split to a CTA (up to 4), two (an odd count leaves the last CTA
one), the largest cluster (16 splits) and partial sums in memory above it."""
import numpy as np
import pytest

import oracle
import workloads as W
from test_gpu_net_output import _inputs
from test_gpu_net_output_x3 import pkg, x3_sigma_rows  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fan_in", [8, 136, 512, 520, 648, 1024, 1032, 1160, 2048, 2056])
def test_splits(pkg, fan_in):  # noqa: F811
    w = W.scaled(W.table2_net(2), widths=(fan_in, 70, 1), acts=(W.ACT_TANH,), dim=fan_in, name=f"k{fan_in}")
    params = W.make_net(w)
    xs = _inputs(w, 131, fan_in)
    with pkg.Mgfwa.for_workload(w, 1, precision=pkg.MGFWA_FP32X3) as run:
        got = run.evaluate(xs, pkg.MGFWA_FP32X3).astype(np.float64)
    ref = oracle.Problem.for_workload(w).fitness_many(xs)
    _, sig = x3_sigma_rows(w, params, xs)
    bad = np.abs(got - ref) > 10.0 * sig + 1e-30
    assert not bad.any(), (fan_in, [(int(i), got[i], ref[i], sig[i]) for i in np.nonzero(bad)[0][:4]])
