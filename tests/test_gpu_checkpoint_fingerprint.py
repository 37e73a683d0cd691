"""A checkpoint's fingerprint is a fixed function of the problem (FNV-1a over the configuration's fields but the budget,
the network and every 61st element of the batch or the parameters), so that checkpoints saved by any build load in any
other: compared here with the same function of the host's arrays."""
import struct

import numpy as np
import pytest

import workloads as W
from test_gpu_checkpoint import pkg  # noqa: F401

pytestmark = pytest.mark.gpu


def fnv(data, f=1469598103934665603):
    for b in data:
        f = ((f ^ b) * 1099511628211) % (1 << 64)
    return f


def expected(cfg, kind, widths, acts, X=None, y=None, params=None):
    names = ["dim", "lb", "ub", "n_fireworks", "sparks_per_firework", "guiding_per_firework", "sigma", "boost",
             "amp_init", "c_amplify", "c_reduce", "seed", "precision", "elite_rescore", "n_runs", "refine_every",
             "refine_steps", "refine_lr", "loser_out", "lagged_guiding", "shard_id", "n_shards"]
    ctype = dict(cfg._fields_)
    data = b"".join(bytes(ctype[n](getattr(cfg, n))) for n in names)
    n_layers = max(len(widths) - 1, 0)
    data += struct.pack("<ii", kind, n_layers)
    if n_layers:
        data += np.asarray(widths, np.int32).tobytes() + np.asarray(acts, np.int32).tobytes()
    if X is not None:
        data += struct.pack("<q", len(X)) + X.ravel()[::61].tobytes() + y[::61].tobytes()
    if params is not None:
        data += params[::61].tobytes()
    return fnv(data)


def saved(h):
    return struct.unpack("<Q", h.checkpoint()[8:16])[0]


@pytest.mark.parametrize("widths, n, precision, kw", [
    ((8, 16, 3), 512, "fp32", {}),
    ((8, 16, 3), 1, "fp32", {"n_runs": 3}),                   # one label, eight inputs
    ((64, 64, 10), 61, "bf16", {"elite_rescore": 1}),
    ((112, 64, 32, 5), 367, "fp8", {"loser_out": 1}),
    ((8, 16, 3), 62, "fp32", {"refine_every": 2, "refine_steps": 1, "refine_lr": 0.25}),
])
def test_mlp(pkg, widths, n, precision, kw):  # noqa: F811
    w = W.scaled(W.MLP_784_64_10, widths=widths, acts=(W.ACT_RELU,) * (len(widths) - 2), n_samples=n, n_fireworks=3,
                 sparks_per_firework=16, guiding_per_firework=4)
    X, y = W.make_data(w)
    prec = {"fp32": pkg.MGFWA_FP32, "bf16": pkg.MGFWA_BF16, "fp8": pkg.MGFWA_FP8}[precision]
    with pkg.Mgfwa.for_workload(w, 21, precision=prec, X=X, y=y, **kw) as h:
        assert saved(h) == expected(h.cfg, pkg.MGFWA_OBJ_MLP_CE, widths, w.acts, X, y)
        h.step(1)
        assert saved(h) == expected(h.cfg, pkg.MGFWA_OBJ_MLP_CE, widths, w.acts, X, y)


def test_net_and_sphere(pkg):  # noqa: F811
    w = W.table2_net(2)
    with pkg.Mgfwa.for_workload(w, 5) as h:
        assert saved(h) == expected(h.cfg, pkg.MGFWA_OBJ_NET_OUTPUT, w.widths, w.acts, params=W.make_net(w))
    with pkg.Mgfwa.for_workload(W.SPHERE_30, 5) as h:
        assert saved(h) == expected(h.cfg, pkg.MGFWA_OBJ_SPHERE, (), ())
