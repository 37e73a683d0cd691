"""The work a user has this library do, as cases that can be timed and compared.

Four kinds of case, each a call a user's program makes:

* ``eval``: the FP32 fitness of spark rows that are already on the GPU
  (``mgfwa_evaluate_fp32_noalloc``), the plain path every lower precision is
  held against.
* ``run``: a whole optimisation: create a handle from host data, run the
  generations of the evaluation budget, read the best position back, destroy.
* ``gradient``: the objective and its gradient (forward and backward) of a
  refining handle's vectors, host vectors in, host gradients out.
* ``group``: many runs of different shapes stepped together, made, run to their
  budgets and read back.

``listed`` holds one case per ordinary use, ``draw`` more of the same ranges.
"""
from __future__ import annotations

import numpy as np
import torch

import paper_2501_03944_gb300 as mg
import workloads as W

ACTS = {"tanh": mg.MGFWA_ACT_TANH, "relu": mg.MGFWA_ACT_RELU, "gelu": mg.MGFWA_ACT_GELU}
PRECISIONS = {"fp32": mg.MGFWA_FP32, "bf16": mg.MGFWA_BF16, "fp8": mg.MGFWA_FP8, "fp32x3": mg.MGFWA_FP32X3}


def listed():
    return [
        # the smallest call: one firework's sparks of the 8-16-3 network, all launch latency
        dict(name="eval_mlp8", kind="eval", widths="8,16,3", act="tanh", data="mixture", n=512, count=40, bound=5.0),
        # one generation's explosion sparks of the bench network on the plain FP32 path
        dict(name="eval_mlp784", kind="eval", widths="784,64,10", act="relu", data="prototypes", n=2048, count=1000,
             bound=1.0),
        # the FP32 leg of the precision sweep's three-layer network: one firework's sparks
        dict(name="eval_mlp3072", kind="eval", widths="3072,128,64,10", act="relu", data="mixture", n=4096,
             count=256, bound=1.0),
        # odd sizes: hidden width, class, sample and spark counts that fill no tile
        dict(name="eval_ragged", kind="eval", widths="200,96,21", act="tanh", data="mixture", n=1003, count=333,
             bound=1.0),
        # plain FP32 run of the 8-16-3 network over its whole budget of 20,000 evaluations
        dict(name="run_mlp8", kind="run", widths="8,16,3", act="tanh", data="mixture", n=512, precision="fp32",
             mu=5, lam=40, m=4, gens=90, bound=5.0, runs=1, loser_out=0, lagged=0),
        # the bench workload: BF16 fitness with the FP32 re-score of the elite
        dict(name="run_mlp784_bf16", kind="run", widths="784,64,10", act="relu", data="prototypes", n=2048,
             precision="bf16", mu=5, lam=200, m=8, gens=50, bound=1.0, runs=1, loser_out=0, lagged=0),
        # the same in FP8, two runs in one handle, with the loser-out tournament
        dict(name="run_mlp784_fp8", kind="run", widths="784,64,10", act="relu", data="prototypes", n=2048,
             precision="fp8", mu=5, lam=200, m=8, gens=25, bound=1.0, runs=2, loser_out=1, lagged=0),
        # the precision sweep's three-layer network in BF16, the largest spark rows
        dict(name="run_mlp3072_bf16", kind="run", widths="3072,128,64,10", act="relu", data="mixture", n=4096,
             precision="bf16", mu=8, lam=256, m=8, gens=10, bound=1.0, runs=1, loser_out=0, lagged=0),
        # the hybrid refinement's forward and backward pass, one vector for each of eight runs
        dict(name="gradient_mlp784", kind="gradient", widths="784,64,10", act="relu", data="prototypes", n=2048,
             runs=8, bound=1.0),
        # the paper's testbed, Table 2's net 10: every layer of all sparks one FP32 product
        dict(name="run_net10", kind="run", widths="1000" + ",512" * 11 + ",1", act="gelu", data="net", n=0,
             precision="fp32", mu=5, lam=200, m=8, gens=20, bound=1.0, runs=1, loser_out=0, lagged=0),
        # the same at FP32 accuracy on the tensor cores, with lagged multi-guiding
        dict(name="run_net10_x3", kind="run", widths="1000" + ",512" * 11 + ",1", act="gelu", data="net", n=0,
             precision="fp32x3", mu=5, lam=200, m=8, gens=20, bound=1.0, runs=1, loser_out=0, lagged=1),
        # many runs of mixed shapes stepped as one graph per generation
        dict(name="group_mixed", kind="group", members=24, shapes=7, gens=10),
    ]


def _odd(rng, lo, hi):
    """A whole number in [lo, hi], spread over its logarithm."""
    return max(lo, min(hi, int(round(float(np.exp(rng.uniform(np.log(lo), np.log(hi))))))))


def draw(rng):
    case = _draw(rng)
    most = max(work(c)["flops"] for c in listed())
    while work(case)["flops"] > most:  # never more than the largest listed case
        case["gens"] = max(1, case["gens"] // 2)
    return case


def _draw(rng):
    kind = rng.choice(["eval", "eval", "run", "run", "run", "gradient", "net", "group"])
    if kind == "eval":
        d_in = 8 * _odd(rng, 1, 384)
        h = rng.choice(["16", "64", "128", "128,64", str(_odd(rng, 4, 192))])
        c = _odd(rng, 2, 32)
        n, count = _odd(rng, 1, 4096), _odd(rng, 1, 1040)
        while d_in * 128.0 * n * count > 3072.0 * 128 * 4096 * 200:
            count = max(1, count // 2)
        return dict(kind="eval", widths=f"{d_in},{h},{c}", act=rng.choice(["tanh", "relu"]),
                    data=rng.choice(["mixture", "prototypes"]), n=n, count=count, bound=rng.choice([1.0, 5.0]))
    if kind == "run":
        net = rng.choice(["mlp8", "two", "two", "three"])
        m = rng.choice([1, 4, 8])
        lam = m * _odd(rng, 4, 256 // m)
        mu = rng.randint(1, 8)
        base = dict(kind="run", mu=mu, lam=lam, m=m, gens=_odd(rng, 1, 20), runs=rng.choice([1, 1, 2]),
                    loser_out=rng.choice([0, 0, 1]), lagged=rng.choice([0, 0, 1]))
        if net == "mlp8":
            return dict(base, widths="8,16,3", act="tanh", data="mixture", n=_odd(rng, 100, 2048), precision="fp32",
                        bound=5.0)
        if net == "two":
            d_in = 16 * _odd(rng, 1, 64)
            return dict(base, widths=f"{d_in},{rng.choice([32, 64, 64, 128])},{_odd(rng, 2, 32)}", act="relu",
                        data="prototypes", n=_odd(rng, 100, 4096), precision=rng.choice(["bf16", "fp8"]), bound=1.0)
        return dict(base, widths=f"{16 * _odd(rng, 8, 192)},128,64,{_odd(rng, 2, 16)}", act="relu", data="mixture",
                    n=_odd(rng, 100, 4096), precision=rng.choice(["bf16", "fp8"]), bound=1.0, gens=_odd(rng, 1, 8),
                    runs=1)
    if kind == "gradient":
        return dict(kind="gradient", widths=f"{8 * _odd(rng, 2, 128)},{rng.choice(['64', '128', '128,64'])}"
                                            f",{_odd(rng, 2, 32)}",
                    act=rng.choice(["tanh", "relu"]), data="prototypes", n=_odd(rng, 100, 4096),
                    runs=_odd(rng, 1, 16), bound=1.0)
    if kind == "net":
        d, h, layers = rng.choice([(10, 16, 5), (20, 32, 5), (100, 64, 8), (200, 128, 8), (1000, 256, 11),
                                   (2000, 512, 11)])
        return dict(kind="run", widths=f"{d}" + f",{h}" * layers + ",1", act=rng.choice(["relu", "gelu"]),
                    data="net", n=0, precision=rng.choice(["fp32", "fp32x3"]), mu=rng.randint(1, 8),
                    lam=8 * _odd(rng, 2, 25), m=8, gens=_odd(rng, 1, 10), bound=1.0, runs=1, loser_out=0,
                    lagged=rng.choice([0, 1]))
    return dict(kind="group", members=rng.randint(2, 24), shapes=rng.randint(0, 1000), gens=rng.randint(2, 10))


# ---------------------------------------------------------------------------
# Inputs.

def _widths(case):
    return tuple(int(v) for v in case["widths"].split(","))


def _acts(case):
    return (ACTS[case["act"]],) * (len(_widths(case)) - 2)


def _batch(case, seed):
    """The shared labelled batch: a Gaussian mixture, or noisy class prototypes in [0, 1]."""
    w, n = _widths(case), case["n"]
    rng = np.random.default_rng([seed, 1])
    d, c = w[0], w[-1]
    y = (np.arange(n) % c).astype(np.int32)
    noise = rng.standard_normal((n, d), dtype=np.float32)
    if case["data"] == "prototypes":
        X = rng.random((c, d), dtype=np.float32)[y] + np.float32(0.1) * noise
        return np.ascontiguousarray(np.clip(X, 0.0, 1.0)), y
    X = rng.standard_normal((c, d), dtype=np.float32)[y] + np.float32(0.5) * noise
    return np.ascontiguousarray(X), y


def _sparks(case, seed, count, dim):
    """Explosion sparks as a generation makes them: five fireworks in the box, each spark within an
    amplitude of its firework, kept inside the bounds (drawn on the GPU)."""
    b = case["bound"]
    g = torch.Generator("cuda").manual_seed(seed)
    fw = torch.empty(5, dim, device="cuda").uniform_(-b, b, generator=g)
    x = torch.empty(count, dim, device="cuda").uniform_(-0.4 * b, 0.4 * b, generator=g)
    return x.add_(fw.repeat(-(-count // 5), 1)[:count]).clamp_(-b, b)


def _network(widths, seed):
    """A testbed network's fixed parameters: each layer U(-1/sqrt(fan_in), 1/sqrt(fan_in))."""
    rng = np.random.default_rng([seed, 2])
    parts = []
    for fi, fo in zip(widths[:-1], widths[1:]):
        parts.append((rng.random(fi * fo + fo, dtype=np.float32) * 2 - 1) / np.float32(np.sqrt(fi)))
    return np.ascontiguousarray(np.concatenate(parts))


def prepare(case, seed):
    kind = case["kind"]
    if kind == "group":
        members = []
        for w in W.mixed_batch(case["members"], case["shapes"], case["gens"]):
            X, y = _batch(dict(widths=",".join(map(str, w.widths)), n=w.n_samples, data="mixture"), seed + w.data_seed)
            members.append((w, mg.MGFWA_FP32 if w.widths[0] == 8 else mg.MGFWA_BF16, X, y))
        return dict(case=case, seed=seed, members=members)
    w = _widths(case)
    state = dict(case=case, seed=seed, widths=w, acts=_acts(case))
    if case["data"] == "net":
        return dict(state, params=_network(w, seed), dim=w[0])
    X, y = _batch(case, seed)
    dim = W.mlp_param_count(w)
    state.update(dim=dim, X=X, y=y)
    if kind == "eval":
        ld = (dim + 3) // 4 * 4
        rows = torch.zeros(case["count"], ld, device="cuda")
        rows[:, :dim] = _sparks(case, seed, case["count"], dim)
        state.update(ld=ld, rows=rows, X_dev=torch.from_numpy(X).cuda(), y_dev=torch.from_numpy(y).cuda(),
                     fit=torch.zeros(case["count"], device="cuda"))
    elif kind == "gradient":
        state["xs"] = _sparks(case, seed, case["runs"], dim).cpu().numpy()
        state["run"] = mg.Mgfwa(dim=dim, lb=-case["bound"], ub=case["bound"], n_fireworks=5, sparks_per_firework=40,
                                guiding_per_firework=4, eval_budget=1 << 40, seed=seed, widths=w, acts=state["acts"],
                                X=X, y=y, n_runs=case["runs"], refine_every=5, refine_steps=10, refine_lr=0.05)
    return state


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "eval":
        mg.mgfwa_evaluate_fp32_noalloc(state["widths"], state["acts"], case["n"], state["X_dev"].data_ptr(),
                                       state["y_dev"].data_ptr(), state["rows"].data_ptr(), state["ld"],
                                       case["count"], state["fit"].data_ptr(),
                                       torch.cuda.current_stream().cuda_stream)
        return state["fit"]
    if kind == "gradient":
        return state["run"].gradient(state["xs"])
    if kind == "group":
        runs = [mg.Mgfwa.for_workload(w, state["seed"] + i, precision=prec, X=X, y=y)
                for i, (w, prec, X, y) in enumerate(state["members"])]
        with mg.Group(runs) as group:
            group.run(case["gens"], chunk=case["gens"])
        best = [r.best() for r in runs]
        for r in runs:
            r.close()
        return (np.concatenate([b[0] for b in best]), np.array([b[1] for b in best]),
                np.array([b[2] for b in best], dtype=np.int64))
    mlp = case["data"] != "net"
    b = case["bound"]
    with mg.Mgfwa(dim=state["dim"], lb=-b, ub=b, n_fireworks=case["mu"], sparks_per_firework=case["lam"],
                  guiding_per_firework=case["m"],
                  eval_budget=W.budget_for_generations(case["mu"], case["lam"], case["m"], case["gens"]),
                  seed=state["seed"], precision=PRECISIONS[case["precision"]],
                  kind=mg.MGFWA_OBJ_MLP_CE if mlp else mg.MGFWA_OBJ_NET_OUTPUT, widths=state["widths"],
                  acts=state["acts"], X=state.get("X"), y=state.get("y"), params=state.get("params"),
                  n_runs=case["runs"], loser_out=case["loser_out"], lagged_guiding=case["lagged"]) as h:
        h.run()
        best = [h.best(r) for r in range(case["runs"])]
    return (np.stack([v[0] for v in best]), np.array([v[1] for v in best]),
            np.array([v[2] for v in best], dtype=np.int64))


# ---------------------------------------------------------------------------
# What a pass cannot do without.

def _mults(w):
    return sum(a * b for a, b in zip(w[:-1], w[1:]))


def _run_work(w, mlp, n, dim, mu, lam, m, gens, runs, data_bytes):
    """Every evaluation's products; the host data read and the best position written once (the sparks in
    between are no output, so their rows are not counted)."""
    evals = runs * (mu + gens * mu * (lam + m))
    flops = 2.0 * _mults(w) * (n if mlp else 1) * evals
    return {"bytes": data_bytes + 4.0 * dim * runs, "flops": flops}


def work(case):
    kind = case["kind"]
    if kind == "group":
        total = {"bytes": 0.0, "flops": 0.0}
        for w in W.mixed_batch(case["members"], case["shapes"], case["gens"]):
            one = _run_work(w.widths, True, w.n_samples, w.dim, w.n_fireworks, w.sparks_per_firework,
                            w.guiding_per_firework, case["gens"], 1, 4.0 * w.n_samples * (w.widths[0] + 1))
            total = {k: total[k] + one[k] for k in total}
        return total
    w, n = _widths(case), case["n"]
    if case["data"] == "net":
        data = 4.0 * W.mlp_param_count(w)
        return _run_work(w, False, 0, w[0], case["mu"], case["lam"], case["m"], case["gens"], case["runs"], data)
    dim = W.mlp_param_count(w)
    data = 4.0 * n * (w[0] + 1)
    if kind == "eval":
        c = case["count"]
        return {"bytes": data + 4.0 * c * (dim + 1), "flops": 2.0 * _mults(w) * n * c}
    if kind == "gradient":
        # forward, weight gradients, and the gradients of the hidden activations
        mults = 2 * _mults(w) + _mults(w[1:])
        return {"bytes": data + 4.0 * case["runs"] * (2 * dim + 1), "flops": 2.0 * mults * n * case["runs"]}
    return _run_work(w, True, n, dim, case["mu"], case["lam"], case["m"], case["gens"], case["runs"], data)


# ---------------------------------------------------------------------------
# The computed values in 64 bits.

def _loss64(x, w, act, X, y):
    """Mean cross-entropy of the flattened parameters `x` in float64."""
    a, off = X, 0
    for l in range(len(w) - 1):
        fi, fo = w[l], w[l + 1]
        Wl = x[off:off + fi * fo].view(fo, fi)
        b = x[off + fi * fo:off + fi * fo + fo]
        off += fi * fo + fo
        a = torch.nn.functional.linear(a, Wl, b)
        if l + 2 < len(w):
            a = torch.tanh(a) if act == "tanh" else torch.relu(a)
    return torch.nn.functional.cross_entropy(a, y)


def exact(case, seed):
    if case["kind"] not in ("eval", "gradient"):
        return None
    w = _widths(case)
    dim = W.mlp_param_count(w)
    X, y = _batch(case, seed)
    X, y = torch.from_numpy(X).cuda().double(), torch.from_numpy(y).cuda().long()
    if case["kind"] == "eval":
        rows = _sparks(case, seed, case["count"], dim)
        return torch.stack([_loss64(r.double(), w, case["act"], X, y) for r in rows])
    f, g = [], []
    for r in _sparks(case, seed, case["runs"], dim):
        x = r.double().requires_grad_(True)
        loss = _loss64(x, w, case["act"], X, y)
        g.append(torch.autograd.grad(loss, x)[0])
        f.append(loss.detach())
    return torch.stack(f), torch.stack(g)
