"""FP32 fitness on the tensor cores: what one spark holds never reaches the fitness of the sparks beside it in a tile."""
import numpy as np
import pytest

import oracle
import workloads as W
from test_gpu_fp32_tc import case, evaluate, pkg  # noqa: F401

pytestmark = pytest.mark.gpu


# 32 sample tiles, so that a tile takes as many sparks as fit its 128 columns: h1 = 8 eight (fewer than the 16 that
# would fit), 17 seven with the fourth across the two halves, 32 four, 43 two with the second across the halves, 64 two
@pytest.mark.parametrize("h1, act", [(8, "relu"), (17, "tanh"), (17, "relu"), (32, "tanh"), (43, "tanh"), (64, "relu")])
def test_operands_that_are_not_finite_stay_in_their_spark(pkg, h1, act):  # noqa: F811
    w, X, y = case((40, h1, 5), act, 4000)
    X = np.abs(X) + 0.1
    xs = W.random_vectors(41, w.dim, -1.0, 1.0, seed=h1)
    clean = evaluate(pkg, w, xs, X, y)
    bad = xs.copy()
    bad[3, 5] = np.inf                              # the first unit
    bad[9, (h1 - 1) * 40 + 7] = -np.inf             # the last unit
    bad[10, 40 * (h1 // 2):40 * h1] = np.nan        # half the units
    bad[40, 39] = np.finfo(np.float32).max          # rounds to a BF16 infinity; the last spark, in a tile not full
    got = evaluate(pkg, w, bad, X, y)
    hit = [3, 9, 10, 40]
    others = [i for i in range(41) if i not in hit]
    assert np.array_equal(got[others], clean[others])
    assert np.array_equal(got, np.concatenate([evaluate(pkg, w, bad[i:i + 1], X, y) for i in range(41)]), equal_nan=True)
    for i in hit:
        if act == "tanh" and i != 10:
            v = bad[i:i + 1].copy()
            v[np.isinf(v)] = np.sign(v[np.isinf(v)]) * 1e30       # saturates as well, with finite sums
            want = oracle.Problem.for_workload(w, X, y).fitness_many(v)[0]
            assert abs(got[i] - want) <= 4e-6 * abs(want)


def test_a_sample_that_is_not_finite(pkg):  # noqa: F811
    """A NaN input makes every spark's loss NaN behind tanh; with ReLU every unit of that sample is max(NaN, 0) = 0, the
    loss of the biases alone, as on the CUDA cores."""
    w, X, y = case((40, 17, 5), "relu", 4000)
    xs = W.random_vectors(20, w.dim, -1.0, 1.0, seed=3)
    X = X.copy()
    X[1234, 7] = np.nan
    got = evaluate(pkg, w, xs, X, y)
    zero = X.copy()
    zero[1234] = 0.0
    flat = xs.copy()
    prob = oracle.Problem.for_workload(w, zero, y)
    want = prob.fitness_many(flat)
    # sample 1234: units max(b1, 0) with the input zeroed against 0 with the NaN
    b1, w2, b2 = xs[:, 680:697].astype(np.float64), xs[:, 697:782].reshape(-1, 5, 17).astype(np.float64), xs[:, 782:787]

    def loss(a):
        z = np.einsum("scj,sj->sc", w2, a) + b2
        return np.log(np.exp(z).sum(1)) - z[:, y[1234]]

    want = want + (loss(np.zeros_like(b1)) - loss(np.maximum(b1, 0.0))) / 4000
    assert np.all(np.abs(got - want) <= 4e-6 * np.abs(want))
