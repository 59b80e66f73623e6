"""The work that users of the pixel array engine have it do, as measurable cases.

Every case goes through the package's public calls (Engine.solve, Engine.batch,
Engine.solve_batch, Engine.contract, Engine.contract_count, CostModel).  A state
holds what a program that makes the call keeps: an Engine, the systems (host
coefficients), output buffers, a planned batch, plotted operands.  The wiring,
resolutions and boxes of a case belong to the case; the coefficients (and the
expressions' constants, the model's samples) come from the seed.

Kinds of case:
  circle     circle and parabola, three variables: the smallest whole solve
  chain      a chain of binary cubics, both ends exposed (matrix products)
  ternary    four ternary cubics, 3-D arrays over shared axes
  butterfly  the paper's 2-D expression system (elementary functions, FP64)
  arrays3d   the paper's 3-D expression system
  chains     many chains planned once and replayed (sub-box sweeps, serving)
  networks   random relation networks planned once and replayed
  fresh      systems seen once: planned, uploaded and solved in one call
  contract   one Boolean cluster of two plotted relations
  count      the same over the counting semiring
  model      the learned join-cost model: predictions, loss and gradients
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1609_00061_gb300 as pa
from paper_1609_00061_gb300 import workloads as W
from paper_1609_00061_gb300.learned import usable_networks

# Resolutions of a batch's variables: multiples of 64, and sizes that are not.
EVEN_RES = [64 * k for k in range(1, 17)]
RAGGED_RES = list(range(51, 1000, 37))

HIDDEN, LAYERS, FEATURES = 128, 3, pa.N_FEATURES  # the cost model as it is trained


def listed():
    return [
        # a small system solved over and over: latency and launches
        {"name": "circle_256", "kind": "circle", "res": 256},
        # the headline workload: 8 plots and 7 Boolean 2048^3 joins
        {"name": "chain8_2048", "kind": "chain", "nrel": 8, "res": 2048},
        # a fine grid whose rows are not whole words and whose row pitch is odd
        {"name": "chain4_4001", "kind": "chain", "nrel": 4, "res": 4001},
        # 3-D arrays, several summed variables
        {"name": "ternary_256", "kind": "ternary", "res": 256},
        # non-polynomial systems at the paper's own size, and on a fine grid
        {"name": "arrays3d_75", "kind": "arrays3d", "res": 75},
        {"name": "butterfly_2048", "kind": "butterfly", "res": 2048},
        # a serving batch of uneven systems, replayed
        {"name": "chains_4096", "kind": "chains", "count": 4096, "shapes": 4, "ragged": False},
        # networks of 12-20 relations, the heaviest joins and layouts
        {"name": "networks_40", "kind": "networks", "count": 40, "shapes": 5},
        # systems that are solved once: host planning counts
        {"name": "fresh_128", "kind": "fresh", "count": 128, "shapes": 9, "ragged": True},
        # one large Boolean cluster
        {"name": "contract_8192", "kind": "contract", "m": 8192, "k": 8192, "n": 8192},
        # solution counts instead of marks
        {"name": "count_2048", "kind": "count", "m": 2048, "k": 2048, "n": 2048},
        # one minibatch of the cost model's training
        {"name": "model_256", "kind": "model", "rows": 256},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["circle", "chain", "chain", "ternary", "butterfly", "arrays3d", "chains",
                       "networks", "networks", "fresh", "contract", "count", "model"])
    if kind == "circle":
        return {"kind": kind, "res": _log_int(rng, 32, 2048)}
    if kind == "chain":
        return {"kind": kind, "nrel": rng.randint(2, 8), "res": _log_int(rng, 64, 4001)}
    if kind == "ternary":
        return {"kind": kind, "res": rng.randint(24, 256)}
    if kind == "butterfly":
        return {"kind": kind, "res": _log_int(rng, 40, 2048)}
    if kind == "arrays3d":
        return {"kind": kind, "res": rng.randint(20, 100)}
    if kind == "chains":
        return {"kind": kind, "count": _log_int(rng, 16, 4096), "shapes": rng.randrange(1 << 20),
                "ragged": rng.random() < 0.5}
    if kind == "networks":
        return {"kind": kind, "count": _log_int(rng, 2, 24), "shapes": rng.randrange(1 << 20)}
    if kind == "fresh":
        return {"kind": kind, "count": _log_int(rng, 4, 128), "shapes": rng.randrange(1 << 20),
                "ragged": rng.random() < 0.5}
    if kind == "model":
        return {"kind": kind, "rows": _log_int(rng, 32, 8192)}
    top = 8192 if kind == "contract" else 4096
    return {"kind": kind, "m": _log_int(rng, 200, top), "k": _log_int(rng, 200, top),
            "n": _log_int(rng, 200, top)}


# ------------------------------------------------------------------ inputs
def _stream(seed):
    return W.SplitMix64(W.SEED_BASE * 7919 + int(seed))


def _recoefficient(systems, seed):
    """The same systems with N(0,1) coefficients from the seed."""
    rng = _stream(seed)
    for sy in systems:
        for r in sy.rels:
            r.coeffs = np.ascontiguousarray(rng.normal(len(r.coeffs)))
    return systems


def _reconstant(system, seed):
    """The same expressions with every constant off by up to one percent."""
    rng = _stream(seed)
    for r in system.rels:
        ops, consts = r.expr
        r.expr = (ops, consts * (0.99 + 0.02 * rng.uniform(len(consts))))
    return system


def _systems(case, seed):
    kind = case["kind"]
    if kind == "circle":
        sy = W.circle_parabola(res=case["res"])
        u = _stream(seed).uniform(3)
        sy.rels[0].coeffs[0] = -(0.8 + 0.4 * u[0]) ** 2     # radius
        sy.rels[1].coeffs[0] = 0.3 + 0.4 * u[1]             # vertex
        sy.rels[1].coeffs[5] = -(0.8 + 0.4 * u[2])          # opening
        return [sy]
    if kind == "chain":
        return _recoefficient([W.chain(res=case["res"], nrel=case["nrel"])], seed)
    if kind == "ternary":
        return _recoefficient([W.ternary(res=case["res"])], seed)
    if kind == "butterfly":
        return [_reconstant(W.butterfly(res=case["res"]), seed)]
    if kind == "arrays3d":
        return [_reconstant(W.arrays_3d(res=case["res"]), seed)]
    if kind in ("chains", "fresh"):
        return _recoefficient(
            W.batched_chains(nsys=case["count"], seed=W.SEED_BASE + case["shapes"],
                             res_choices=RAGGED_RES if case["ragged"] else EVEN_RES), seed)
    if kind == "networks":
        nets = usable_networks(W.random_networks(case["count"], seed=W.SEED_BASE + case["shapes"]))
        if not nets:
            nets = [W.chain(res=256, nrel=6)]
        return _recoefficient(nets, seed)
    raise ValueError(kind)


def _pair(case, seed):
    """Axes and two binary cubics R1(v0, v1), R2(v1, v2) on [-3, 3)."""
    axes = [(-3.0, 3.0, case["m"]), (-3.0, 3.0, case["k"]), (-3.0, 3.0, case["n"])]
    rng = _stream(seed)
    return axes, [W.Relation((0, 1), 3, W.random_cubic(rng, 2)),
                  W.Relation((1, 2), 3, W.random_cubic(rng, 2))]


def _words(sy):
    return pa.pa_array_words([sy.axes[v][2] for v in sy.exposed])


def _outputs(systems):
    """One buffer for the results of many systems, each at a 256-byte boundary."""
    sizes = [(_words(sy) + 31) // 32 * 32 for sy in systems]
    buf = torch.zeros(sum(sizes), dtype=torch.int64, device="cuda:0")
    outs, at = [], 0
    for sy, n in zip(systems, sizes):
        outs.append(pa.BitArray(buf[at:at + _words(sy)], tuple(sy.exposed),
                                tuple(sy.axes[v][2] for v in sy.exposed)))
        at += n
    return buf, outs


def _layer_sizes():
    return [FEATURES] + [HIDDEN] * LAYERS + [1]


def _model_inputs(case, seed):
    """Parameters (per layer weights [out][in], then biases), samples and targets."""
    rng = np.random.default_rng(int(seed))
    sizes = _layer_sizes()
    parts = []
    for ni, no in zip(sizes[:-1], sizes[1:]):
        lim = math.sqrt(6.0 / ni)
        parts.append(rng.uniform(-lim, lim, no * ni))
        parts.append(rng.uniform(-0.1, 0.1, no))
    x = rng.uniform(0.0, 1.0, (case["rows"], FEATURES))
    x[:, 15] = 1.0
    t = rng.uniform(0.2, 1.6, case["rows"])
    return [a.astype(np.float32) for a in (np.concatenate(parts), x, t)]


def prepare(case, seed):
    kind = case["kind"]
    eng = pa.Engine(0)
    state = {"kind": kind, "engine": eng}
    if kind in ("contract", "count"):
        axes, rels = _pair(case, seed)
        state["a"] = eng.plot(rels[0], axes)
        state["b"] = eng.plot(rels[1], axes)
    elif kind == "model":
        p, x, t = _model_inputs(case, seed)
        model = pa.CostModel(eng, hidden=HIDDEN, nlayers=LAYERS)
        model.set_params(p)
        state.update(model=model, x=torch.from_numpy(x).cuda(), t=torch.from_numpy(t).cuda())
    else:
        systems = _systems(case, seed)
        buf, outs = _outputs(systems)
        state.update(systems=systems, buf=buf, outs=outs)
        if kind in ("chains", "networks"):
            state["batch"] = eng.batch(systems, outs=outs)
    return state


def run(state):
    kind, eng = state["kind"], state["engine"]
    if kind in ("chains", "networks"):
        state["batch"].run()
        return state["buf"]
    if kind == "fresh":
        eng.solve_batch(state["systems"], outs=state["outs"])
        return state["buf"]
    if kind == "contract":
        return eng.contract(state["a"], state["b"], (0, 2)).words
    if kind == "count":
        return eng.contract_count(state["a"], state["b"], (0, 2))
    if kind == "model":
        model = state["model"]
        y = model.forward(state["x"])
        loss = model.backward(state["x"], state["t"])
        return {"y": y, "loss": loss, "grads": model.get_grads()}
    eng.solve(state["systems"][0], out=state["outs"][0])
    return state["buf"]


def work(case):
    """Inputs read and outputs written once.  Plots: every pixel centre's
    polynomial takes its degree in multiply-adds, every expression its
    operations; counts: every multiply-add of the cluster; the Boolean products
    are not counted (how much of one can be skipped depends on the plots)."""
    kind = case["kind"]
    if kind in ("contract", "count"):
        m, k, n = case["m"], case["k"], case["n"]
        read = 8 * (m * ((k + 63) // 64) + k * ((n + 63) // 64))
        if kind == "count":
            return {"bytes": read + 4 * m * n, "flops": 2.0 * m * k * n}
        return {"bytes": read + 8 * m * ((n + 63) // 64), "flops": 0.0}
    if kind == "model":
        sizes, n = _layer_sizes(), case["rows"]
        weights = sum(a * b for a, b in zip(sizes[:-1], sizes[1:]))
        params = weights + sum(sizes[1:])
        # a forward pass for the predictions; forward, weight and input
        # gradients (not those of the samples) for the step
        macs = n * (4 * weights - FEATURES * HIDDEN)
        return {"bytes": 4.0 * (2 * params + n * (FEATURES + 2)), "flops": 2.0 * macs}
    nbytes = flops = 0.0
    for sy in _systems(case, 0):
        nbytes += 8 * _words(sy)
        for r in sy.rels:
            pixels = math.prod(sy.axes[v][2] for v in set(r.vars))
            if r.expr is None:
                nbytes += 8 * len(r.coeffs)
                flops += 2.0 * r.degree * pixels
            else:
                nbytes += 4 * len(r.expr[0]) + 8 * len(r.expr[1])
                flops += float(sum(1 for o in r.expr[0] if (int(o) & 0xff) > W.X_VAR)) * pixels
    return {"bytes": nbytes, "flops": flops}


def exact(case, seed):
    """The cost model's predictions, loss and gradients in 64 bits; every other
    output is whole numbers."""
    if case["kind"] != "model":
        return None
    p, x, t = (a.astype(np.float64) for a in _model_inputs(case, seed))
    sizes = _layer_sizes()
    layers, at = [], 0
    for ni, no in zip(sizes[:-1], sizes[1:]):
        layers.append((p[at:at + no * ni].reshape(no, ni), p[at + no * ni:at + no * ni + no]))
        at += no * ni + no
    acts = [x]
    for i, (w, b) in enumerate(layers):
        z = acts[-1] @ w.T + b
        acts.append(np.maximum(z, 0.0) if i + 1 < len(layers) else z)
    y = acts[-1][:, 0]
    loss = 0.5 * float(np.mean((y - t) ** 2))
    d = ((y - t) / len(t))[:, None]
    grads = []
    for i in range(len(layers) - 1, -1, -1):
        grads[:0] = [(d.T @ acts[i]).reshape(-1), d.sum(axis=0)]
        if i:
            d = (d @ layers[i][0]) * (acts[i] > 0)
    return {"y": y, "loss": loss, "grads": np.concatenate(grads)}
