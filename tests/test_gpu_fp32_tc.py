"""FP32 fitness with the first layer on the tensor cores (mgfwa_evaluate_fp32_noalloc's path for networks of a
million first-layer products a spark up): sizes at the edges of its tiles, and operands that are not finite."""
import numpy as np
import pytest

import oracle
import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2501_03944_gb300 as p
    return p


ACT = {"tanh": W.ACT_TANH, "relu": W.ACT_RELU}


def evaluate(pkg, w, xs, X, y):
    import torch
    ld = (w.dim + 3) // 4 * 4
    rows = torch.zeros(len(xs), ld, device="cuda")
    rows[:, :w.dim] = torch.from_numpy(xs).cuda()
    Xd, yd = torch.from_numpy(X).cuda(), torch.from_numpy(y).cuda()
    fit = torch.zeros(len(xs), device="cuda")
    pkg.mgfwa_evaluate_fp32_noalloc(w.widths, w.acts, w.n_samples, Xd.data_ptr(), yd.data_ptr(), rows.data_ptr(), ld,
                                    len(xs), fit.data_ptr(), torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    return fit.cpu().numpy()


def case(widths, act, n):
    w = W.scaled(W.MLP_784_64_10, widths=widths, acts=(ACT[act],) * (len(widths) - 2), n_samples=n)
    X, y = W.make_data(w)
    return w, X, y


# FP32 parity's usual 1e-4 would pass a 16-bit product; the sums here are FP32-accurate, so 4e-6: 32 units in the
# last place of the loss, for sums of up to 3072 rounded products averaged over the batch.
@pytest.mark.parametrize("widths, act, n, count", [
    ((16, 8, 2), "relu", 8193, 1), ((40, 64, 10), "tanh", 640, 3), ((56, 17, 5), "relu", 1153, 9),
    ((72, 43, 32), "tanh", 383, 5), ((64, 65, 4), "relu", 257, 2), ((200, 96, 21), "tanh", 333, 7),
    ((784, 64, 10), "relu", 300, 5), ((96, 128, 32), "relu", 130, 4), ((64, 128, 64, 10), "relu", 200, 3),
    ((88, 30, 7, 3), "tanh", 511, 11), ((32, 64, 33, 16), "relu", 513, 6), ((3072, 128, 64, 10), "relu", 3, 2)])
def test_matches_the_oracle_at_tile_edges(pkg, widths, act, n, count):
    w, X, y = case(widths, act, n)
    xs = W.random_vectors(count, w.dim, -1.0, 1.0, seed=5)
    want = oracle.Problem.for_workload(w, X, y).fitness_many(xs)
    got = evaluate(pkg, w, xs, X, y).astype(np.float64)
    assert np.all(np.abs(got - want) <= 4e-6 * np.abs(want) + 1e-7), (got, want)


def test_operands_that_are_not_finite(pkg):
    """An infinite weight behind a saturating activation leaves a finite loss, a NaN weight behind tanh does not, and
    neither reaches the sparks that share the tile."""
    w, X, y = case((64, 64, 10), "tanh", 300)
    X = np.abs(X) + 0.1                                   # the infinite weight's products all have one sign
    xs = W.random_vectors(4, w.dim, -1.0, 1.0, seed=6)
    clean = evaluate(pkg, w, xs, X, y)
    bad = xs.copy()
    bad[1, 5] = np.inf                                    # W1[0][5]: unit 0 saturates at tanh(inf) = 1
    bad[2, 64 + 9] = np.nan
    got = evaluate(pkg, w, bad, X, y)
    assert got[0] == clean[0] and got[3] == clean[3]
    assert np.isnan(got[2])
    big = xs[1:2].copy()
    big[0, 5] = 1e30                                      # saturates as well, with finite sums
    want = oracle.Problem.for_workload(w, X, y).fitness_many(big)[0]
    assert abs(got[1] - want) <= 4e-6 * abs(want)
