"""The testbed's FP32 layers in every tile (64 x 64, 64 x 32, 32 x 32 and 8 x 32 outputs, by how many of them there are
for the SMs) with 16-byte copies and, where a fan-in or a row stride is not a multiple of four, 4-byte ones: a row's value
is bitwise the same in all of them, and the oracle's within the rounding model of tests/test_gpu_net_output.py."""
import numpy as np
import pytest

import oracle
import workloads as W
from test_gpu_net_output import _inputs, fp32_sigma_rows, pkg  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("widths, rows", [
    ((203, 451, 1), 1040),        # 64 x 64 tiles, 4-byte copies; ragged rows, columns and fan-in
    ((204, 452, 1), 1040),        # the same with 16-byte copies
    ((203, 301, 1), 1040),        # 64 x 32
    ((204, 300, 1), 1000),
    ((203, 317, 1), 500),         # 32 x 32
    ((212, 316, 1), 491),
    ((203, 451, 449, 1), 1033),   # the second layer's input rows 451 floats apart
    ((16, 450, 450, 1), 1040),    # one 16-wide chunk; a fan-in that is no multiple of four
])
def test_a_rows_value_is_the_same_in_every_tile(pkg, widths, rows):  # noqa: F811
    w = W.scaled(W.table2_net(10), widths=widths, acts=(W.ACT_GELU,) * (len(widths) - 2), dim=widths[0],
                 name="x".join(map(str, widths)))
    xs = _inputs(w, rows, 17)
    with pkg.Mgfwa.for_workload(w, 1) as run:
        full = run.evaluate(xs)
        some = np.r_[0:40, rows - 7:rows]                     # 8-row tiles
        few = run.evaluate(xs[some])
        one = run.evaluate(xs[rows - 1:])
    assert np.array_equal(full[some], few) and full[-1] == one[0]
    ref = oracle.Problem.for_workload(w).fitness_many(xs)
    assert np.all(np.abs(full - ref) <= 1e-4 * (np.abs(ref) + 1e-2))
    _, sig = fp32_sigma_rows(w, W.make_net(w), xs[some])
    bad = np.abs(full[some].astype(np.float64) - ref[some]) > 10.0 * sig + 1e-30
    assert not bad.any(), (widths, np.nonzero(bad)[0][:4])
