"""A bounded wait that runs out in the FP32 first layer on the tensor cores and in the FP32X3 layers, as
tests/test_gpu_timeout.py does it for the low precisions: with a budget of a few ticks an ordinary wait gives up, the
call reports it, and the handle then works as before.  Nothing faults and no arrival is withheld."""
import numpy as np
import pytest

import workloads as W
from test_gpu_timeout import pkg  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("widths", [(784, 64, 10), (64, 128, 64, 5), (200, 17, 3)])
def test_fp32_first_layer(pkg, widths):  # noqa: F811
    w = W.scaled(W.MLP_784_64_10, widths=widths, acts=(W.ACT_RELU,) * (len(widths) - 2), n_samples=700, n_fireworks=2,
                 sparks_per_firework=12, guiding_per_firework=2)
    X, y = W.make_data(w)
    xs = W.random_vectors(24, w.dim, -1.0, 1.0, seed=9)
    with pkg.Mgfwa.for_workload(w, 3, precision=pkg.MGFWA_FP32, X=X, y=y) as run:
        ref = run.evaluate(xs, pkg.MGFWA_FP32)
        run.wait_budget(16)
        with pytest.raises(pkg.MgfwaError) as e:
            run.evaluate(xs, pkg.MGFWA_FP32)
        assert e.value.status == pkg.MGFWA_ETIMEOUT
        run.wait_budget(0)
        assert np.array_equal(run.evaluate(xs, pkg.MGFWA_FP32), ref)
        assert run.step(2) == pkg.MGFWA_OK
    with pkg.Mgfwa.for_workload(w, 3, precision=pkg.MGFWA_FP32, X=X, y=y) as run2:
        assert np.array_equal(run2.evaluate(xs, pkg.MGFWA_FP32), ref)


@pytest.mark.parametrize("fan_in", [128, 1000, 2056])  # one split to a CTA, two, partial sums in memory
def test_fp32x3_layers(pkg, fan_in):  # noqa: F811
    w = W.scaled(W.table2_net(2), widths=(fan_in, 64, 1), acts=(W.ACT_TANH,), dim=fan_in, name=f"k{fan_in}")
    xs = W.random_vectors(131, fan_in, -1.0, 1.0, seed=9)
    with pkg.Mgfwa.for_workload(w, 1, precision=pkg.MGFWA_FP32X3) as run:
        ref = run.evaluate(xs, pkg.MGFWA_FP32X3)
        run.wait_budget(16)
        with pytest.raises(pkg.MgfwaError) as e:
            run.evaluate(xs, pkg.MGFWA_FP32X3)
        assert e.value.status == pkg.MGFWA_ETIMEOUT
        run.wait_budget(0)
        assert np.array_equal(run.evaluate(xs, pkg.MGFWA_FP32X3), ref)
