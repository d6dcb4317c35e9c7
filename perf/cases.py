"""The work that a user of the counter has it do, as cases that can be timed and compared.

A case names an entry point (`kind`) and a problem: a `family` of network, box and property,
the network's sizes, and how much of it (`depth`, `n` boxes, `problems`).  `prepare` makes the
problem from a seed and loads it into a context, `run` is one call sequence of a user's program.
Networks are seeded (weights N(0, 2/fan_in), biases N(0, 0.1)); where a property could be
trivially safe or unsafe, the draw is repeated until a sampled violation rate lies in a window.
"""
from __future__ import annotations

import math
from types import SimpleNamespace

import numpy as np
import torch

from paper_2312_05890_gb300 import Counter


def listed():
    return [
        # A whole count of a very small network: many levels of few boxes, so the latency of a level counts.
        dict(name="count_tiny", kind="count", family="square", d=2, width=8, hidden=2, out=1, act="relu", depth=16),
        # The collision-avoidance shape at full depth: the main use, millions of boxes on the fused tile kernel.
        dict(name="count_collision", kind="count", family="collision", d=5, width=50, hidden=6, out=5, act="relu",
             depth=20),
        # The mapless-navigation shape: many inputs, two layers; hardly any box is decided, so every level doubles.
        dict(name="count_navigation", kind="count", family="navigation", d=22, width=64, hidden=2, out=3, act="relu",
             depth=18),
        # An image classifier: the state of a box is in HBM and every layer is a matrix product.
        dict(name="count_image", kind="count", family="image", d=784, width=256, hidden=3, out=10, act="relu",
             depth=12),
        # The other activations: the collision-avoidance shape with tanh.
        dict(name="count_collision_tanh", kind="count", family="collision", d=5, width=50, hidden=6, out=5,
             act="tanh", depth=16),
        # Many properties of networks of uneven sizes in one call.
        dict(name="count_batch", kind="batch", problems=48, networks=12, width=64, depth_lo=8, depth_hi=15),
        # Bounds of a handful of boxes, as a program asks for while it looks at single regions: latency.
        dict(name="bounds_navigation_few", kind="bounds", family="navigation", d=22, width=64, hidden=2, out=3, n=64),
        # Bounds of many boxes of the caller's own (another splitting rule, a reachability tool).
        dict(name="bounds_collision_many", kind="bounds", family="collision", d=5, width=50, hidden=6, out=5,
             n=200001),
        # Bounds of perturbed images, one box each.
        dict(name="bounds_image", kind="bounds", family="image", d=784, width=256, hidden=3, out=10, n=1000),
        # The backward pass of a certified training step: gradients of the weights, biases and boxes.
        dict(name="backward_collision", kind="backward", family="collision", d=5, width=50, hidden=6, out=5, n=8192,
             weights=True, slopes=False),
        # Gradients of the lower slopes and the boxes of an image classifier, at supplied slopes.
        dict(name="backward_image", kind="backward", family="image", d=784, width=256, hidden=3, out=10, n=256,
             weights=False, slopes=True),
        # Twenty projected-Adam steps on the lower slopes of undecided boxes.
        dict(name="optimise_collision", kind="optimise", family="collision", d=5, width=50, hidden=6, out=5, n=4096,
             steps=20),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["count", "count", "count", "batch", "bounds", "bounds", "backward", "optimise"])
    if kind == "batch":
        # (a batch's networks are at most as wide as its cost allows)
        return dict(kind="batch", problems=_log_int(rng, 4, 48), networks=rng.randint(1, 12),
                    width=rng.choice([32, 64]), depth_lo=8, depth_hi=rng.randint(9, 14))
    family = rng.choice(["square", "collision", "collision", "navigation", "image"])
    if family == "square":
        net = dict(d=rng.randint(2, 3), width=rng.randint(6, 32), hidden=rng.randint(1, 3), out=1)
    elif family == "collision":
        net = dict(d=5, width=rng.randint(17, 64), hidden=rng.randint(2, 7), out=rng.randint(3, 6))
    elif family == "navigation":
        net = dict(d=rng.randint(9, 32), width=rng.randint(24, 96), hidden=rng.randint(1, 3), out=rng.randint(3, 5))
    else:
        net = dict(d=rng.randint(144, 784), width=rng.randint(48, 256), hidden=rng.randint(2, 3), out=10)
    case = dict(kind=kind, family=family, **net)
    per_box = _flops_per_box(case)
    if kind == "count":
        # the depth that keeps a count of 2^(depth + 1) boxes below the largest listed one
        most = {"square": 18, "collision": 20, "navigation": 17, "image": 11}[family]
        limit = {"square": 1e12, "collision": 6e11, "navigation": 1e11, "image": 1.5e12}[family]
        depth = min(most, int(math.log2(limit / per_box)) - 1)
        act = rng.choice(["relu", "relu", "relu", "tanh", "sigmoid"]) if family in ("square", "collision") else "relu"
        return dict(case, act=act, depth=rng.randint(max(4, depth - 7), depth))
    most = {"square": 100000, "collision": 50000, "navigation": 20000, "image": 500}[family]
    if kind == "bounds":
        return dict(case, n=_log_int(rng, 1, most))
    if kind == "backward":
        weights = family != "image" and rng.random() < 0.5
        return dict(case, n=_log_int(rng, 1, most // 8), weights=weights, slopes=rng.random() < 0.5)
    return dict(case, n=_log_int(rng, 1, most // 32), steps=rng.randint(1, 20))


# ---- problems -------------------------------------------------------------------------------


def _widths(case):
    return [case["d"]] + [case["width"]] * case["hidden"] + [case["out"]]


def _mlp(rng, widths, act="relu"):
    W, b = [], []
    for n_in, n_out in zip(widths[:-1], widths[1:]):
        W.append(rng.normal(0.0, math.sqrt(2.0 / n_in), size=(n_out, n_in)).astype(np.float32))
        b.append(rng.normal(0.0, math.sqrt(0.1), size=n_out).astype(np.float32))
    return SimpleNamespace(W=W, b=b, act=[act] * (len(W) - 1) if act != "relu" else [])


def _values(net, x):
    act = {"tanh": np.tanh, "sigmoid": lambda z: 1.0 / (1.0 + np.exp(-z))}.get(
        net.act[0] if net.act else "", lambda z: np.maximum(z, 0.0))
    h = x.astype(np.float32)
    for k, (w, b) in enumerate(zip(net.W, net.b)):
        h = h @ w.T + b
        if k + 1 < len(net.W):
            h = act(h)
    return h


def _property(clauses):
    rows = [r for clause in clauses for r in clause]
    return SimpleNamespace(rows_per_clause=np.array([len(c) for c in clauses], dtype=np.int32),
                           C=np.array([r[0] for r in rows], dtype=np.float32),
                           e=np.array([r[1] for r in rows], dtype=np.float32),
                           strict=np.array([r[2] for r in rows], dtype=np.uint8))


def _rate(rng, net, lo, hi, prop, samples=4096):
    """The sampled share of the box that violates the property."""
    x = lo + (hi - lo) * rng.random((samples, lo.size), dtype=np.float32)
    v = _values(net, x) @ prop.C.T + prop.e
    ok = np.where(prop.strict.astype(bool), v > 0, v >= 0)
    bad, r0 = np.zeros(len(x), dtype=bool), 0
    for nr in prop.rows_per_clause:
        bad |= ok[:, r0:r0 + nr].all(axis=1)
        r0 += nr
    return float(bad.mean())


def _minus(n, i, j, scale_i=1.0, scale_j=1.0):
    c = np.zeros(n, dtype=np.float32)
    c[i], c[j] = scale_i, -scale_j
    return c


def _problem(case, rng):
    """Network, box and unsafe set of one seeded problem of the case's family."""
    family, d, out = case["family"], case["d"], case["out"]
    while True:
        net = _mlp(rng, _widths(case), case.get("act", "relu"))
        if family == "square":        # [-1, 1]^d, unsafe where the output is negative
            lo, hi, window = np.full(d, -1.0), np.full(d, 1.0), (0.05, 0.95)
            prop = _property([[(np.full(1, -1.0), 0.0, True)]])
        elif family == "collision":   # unsafe where output 0 is not the least
            side = rng.uniform(0.05, 0.3, size=d)
            lo = rng.uniform(-0.5, 0.5 - side)
            hi, window = lo + side, (0.005, 0.5)
            prop = _property([[(_minus(out, 0, j), 0.0, True)] for j in range(1, out)])
        elif family == "navigation":  # unsafe where action 1 is chosen
            c = np.concatenate([rng.uniform(0.025, 0.975, size=d - 2), rng.uniform(-0.995, 0.995, size=2)])
            half = np.array([0.025] * (d - 2) + [0.005] * 2)
            lo, hi, window = c - half, c + half, (0.05, 0.5)
            prop = _property([[(_minus(out, 1, j), 0.0, False) for j in range(out) if j != 1]])
        else:                         # image: class 0 stays on top around a point it is on top at
            x0 = rng.random(d)
            top = int(np.argmax(_values(net, x0[None])[0]))
            for a in (net.W[-1], net.b[-1]):
                a[[0, top]] = a[[top, 0]]
            lo, hi, window = np.clip(x0 - 0.02, 0.0, 1.0), np.clip(x0 + 0.02, 0.0, 1.0), None
            prop = _property([[(_minus(out, j, 0), 0.0, False)] for j in range(1, out)])
        lo, hi = lo.astype(np.float32), hi.astype(np.float32)
        if window is None or window[0] <= _rate(rng, net, lo, hi, prop) <= window[1]:
            return SimpleNamespace(net=net, lo=lo, hi=hi, prop=prop)


def _batch(case, rng):
    """Problems of uneven size: several boxes and one-clause properties for each of some networks."""
    problems = []
    dims = [5, 8, 16, 5]
    for k in range(case["networks"]):
        d = dims[k % len(dims)]
        want = (k + 1) * case["problems"] // case["networks"]
        tries = 0
        while len(problems) < want:
            if tries % 16 == 0:   # a network whose outputs lie too far apart for such rows is drawn again
                width, hidden = int(rng.choice([32, case["width"]])), int(rng.integers(2, 7))
                net = _mlp(rng, [d] + [width] * hidden + [int(rng.integers(2, 9))])
            tries += 1
            side = rng.uniform(0.02, 0.2, size=d)
            lo = rng.uniform(-0.5, 0.5 - side).astype(np.float32)
            hi = (lo + side).astype(np.float32)
            rows, n_out = [], len(net.b[-1])
            for _ in range(int(rng.integers(1, 3))):
                i, j = rng.choice(n_out, size=2, replace=False)
                rows.append((_minus(n_out, i, j, rng.uniform(0.5, 2.0), rng.uniform(0.5, 2.0)),
                             rng.normal(0.0, math.sqrt(0.1)), False))
            prop = _property([rows])
            if 0.01 <= _rate(rng, net, lo, hi, prop, 512) <= 0.99:
                depth = case["depth_lo"] + 5 * len(problems) % (case["depth_hi"] - case["depth_lo"] + 1)
                problems.append(SimpleNamespace(net=net, lo=lo, hi=hi, prop=prop, depth=depth))
    return problems


def _sub_boxes(p, n, rng):
    """Boxes inside the problem's box, each side a half to a sixteenth of it and finer, as bisection makes them."""
    w = p.hi - p.lo
    side = w * np.exp2(-rng.uniform(1.0, 5.0, size=(n, p.lo.size)))
    lo = p.lo + (w - side) * rng.random((n, p.lo.size))
    return lo.astype(np.float32), (lo + side).astype(np.float32)


def _inputs(case, seed):
    """Everything that a pass reads, on the host."""
    rng = np.random.default_rng(seed)
    if case["kind"] == "batch":
        return SimpleNamespace(problems=_batch(case, rng))
    p = _problem(case, rng)
    s = SimpleNamespace(p=p, alpha=None)
    if "n" in case:
        s.lo, s.hi = _sub_boxes(p, case["n"], rng)
    if case["kind"] == "backward":
        rows = p.prop.e.size
        s.g_lo = rng.normal(size=(case["n"], rows)).astype(np.float32)
        s.g_hi = rng.normal(size=(case["n"], rows)).astype(np.float32)
        if case["slopes"]:
            s.alpha = rng.random((case["n"], case["width"] * case["hidden"]), dtype=np.float32)
    return s


def prepare(case, seed):
    s = _inputs(case, seed)
    s.case = case
    s.counter = Counter(0)
    if case["kind"] == "batch":
        return s
    s.counter.set_problem(s.p)
    for name in ("lo", "hi", "g_lo", "g_hi", "alpha"):
        if getattr(s, name, None) is not None:
            setattr(s, name, torch.from_numpy(getattr(s, name)).cuda())
    return s


# ---- one pass -------------------------------------------------------------------------------


def _count_outputs(res):
    """What a count says (its timings and internal tallies are not results)."""
    out = {k: res[k] for k in ("unsafe_lo", "unsafe_hi", "boxes", "tie_leaves")}
    for k in ("level_boxes", "level_safe", "level_unsafe", "level_undecided"):
        out[k] = np.array(res[k], dtype=np.int64)
    return out


def run(state):
    case, c = state.case, state.counter
    if case["kind"] == "count":
        # one query of a verification session: the network stays, box and property are the query's
        p = state.p
        c.set_box(p.lo, p.hi)
        c.set_property(p.prop.rows_per_clause, p.prop.C, p.prop.e, p.prop.strict)
        out = _count_outputs(c.count(case["depth"]))
        out["schedule"] = c.schedule(case["depth"])   # which input each level halved: the codes' meaning
        return out
    if case["kind"] == "batch":
        res = [_count_outputs(r) for r in c.count_batch(state.problems)]
        return {k: np.concatenate([np.atleast_1d(r[k]) for r in res]) for k in res[0]}
    if case["kind"] == "bounds":
        lo, hi, _ = c.bounds(state.lo, state.hi, want_cls=False)
        return {"row_lo": lo, "row_hi": hi}
    if case["kind"] == "backward":
        return c.margin_backward(state.lo, state.hi, state.g_lo, state.g_hi, alpha=state.alpha,
                                 weights=case["weights"])
    lo, hi, cls, alpha = c.optimize_alpha(state.lo, state.hi, steps=case["steps"])
    return {"row_lo": lo, "row_hi": hi, "cls": cls, "alpha": alpha}


# ---- the work of a pass -----------------------------------------------------------------------


def _flops_per_box(case):
    """The contractions of both equations of every neuron: centre and radius products over d + 1 columns."""
    w = _widths(case)
    return 4.0 * (case["d"] + 1) * sum(a * b for a, b in zip(w[1:-1], w[2:])) + 4.0 * case["d"] * w[1]


def _boxes(d, depth):
    """Boxes of a count: a level doubles until the undecided boxes are those at the boundary of the unsafe set."""
    if d <= 3:
        return 2.0 * sum(2.0 ** (t * (d - 1) / d) for t in range(depth + 1))
    return 2.0 ** (depth + 1) - 1


def work(case):
    if case["kind"] == "batch":
        per = _flops_per_box(dict(d=8, width=(32 + case["width"]) / 2, hidden=4, out=2))
        depths = range(case["depth_lo"], case["depth_hi"] + 1)
        boxes = case["problems"] * sum(_boxes(8, t) for t in depths) / len(depths)
        return {"bytes": 25.0 * boxes, "flops": per * boxes}
    w = _widths(case)
    params = 4.0 * sum(a * b + b for a, b in zip(w[:-1], w[1:]))
    per = _flops_per_box(case)
    if case["kind"] == "count":
        # per box its path code read and its class written, and two children's codes written
        boxes = _boxes(case["d"], case["depth"])
        return {"bytes": params + 25.0 * boxes, "flops": per * boxes}
    n, d = case["n"], case["d"]
    rows = {"square": 1, "collision": case["out"] - 1, "navigation": case["out"] - 1, "image": 9}[case["family"]]
    hidden = case["width"] * case["hidden"]
    if case["kind"] == "bounds":
        return {"bytes": params + 4.0 * n * (2 * d + 2 * rows), "flops": per * n}
    if case["kind"] == "backward":
        moved = 4.0 * n * (4 * d + 4 * rows + hidden * (2 if case["slopes"] else 1))
        return {"bytes": params * (2 if case["weights"] else 1) + moved,
                "flops": per * n * (3 if case["weights"] else 2)}
    return {"bytes": params + 4.0 * n * (2 * d + 2 * rows + hidden) + n, "flops": 3 * per * n * case["steps"]}


# ---- the same outputs in 64 bits --------------------------------------------------------------


def _row_bounds64(W, b, C, e, lo, hi, alpha):
    """Row bounds of boxes by symbolic linear relaxation, and the lower slopes used (n x neurons)."""
    m, r = (lo + hi) / 2, (hi - lo) / 2
    W, b = list(W), list(b)
    W[-1], b[-1] = C @ W[-1], C @ b[-1] + e
    upper = torch.cat([W[0] * r[:, None, :], (m @ W[0].T + b[0])[:, :, None]], dim=2)
    lower, slopes = upper, []
    for k in range(1, len(W)):
        su, sl = upper[..., :-1].abs().sum(-1), lower[..., :-1].abs().sum(-1)
        ll, ul = lower[..., -1] - sl, lower[..., -1] + sl
        lu, uu = upper[..., -1] - su, upper[..., -1] + su
        on, off = ll >= 0, (uu <= 0) & (ll < 0)
        chord = ~on & ~off & (lu < 0)
        up = torch.where(chord, uu / torch.where(chord, uu - lu, 1.0), 1.0)
        sloped = ~on & ~off & (ul > 0)
        if alpha is None:
            a = torch.where(sloped, ul / torch.where(sloped, ul - ll, 1.0), 0.0)
        else:
            at = sum(s.shape[1] for s in slopes)
            a = alpha[:, at:at + ll.shape[1]].clamp(0, 1)
        if a.requires_grad:
            a.retain_grad()
        slopes.append(a)
        shift = torch.cat([torch.zeros_like(upper[..., :-1]), torch.where(chord, lu, 0.0)[..., None]], dim=-1)
        up = torch.where(off, 0.0, up)
        low = torch.where(on, 1.0, torch.where(sloped, a, 0.0))
        upper, lower = up[..., None] * (upper - shift), low[..., None] * lower
        centre, radius = W[k] @ ((upper + lower) / 2), W[k].abs() @ ((upper - lower) / 2)
        centre = torch.cat([centre[..., :-1], centre[..., -1:] + b[k][:, None]], dim=-1)
        upper, lower = centre + radius, centre - radius
    return (lower[..., -1] - lower[..., :-1].abs().sum(-1), upper[..., -1] + upper[..., :-1].abs().sum(-1), slopes)


def exact(case, seed):
    if case["kind"] not in ("bounds", "backward"):
        # counts are whole numbers; a slope that Adam moves by the sign of its gradient has no 64-bit value to meet
        return None
    s = _inputs(case, seed)
    grad = case["kind"] == "backward"

    def t64(a, leaf=False):
        return torch.from_numpy(np.asarray(a)).cuda().double().requires_grad_(leaf)

    W = [t64(w, grad and case["weights"]) for w in s.p.net.W]
    b = [t64(x, grad and case["weights"]) for x in s.p.net.b]
    C, e = t64(s.p.prop.C), t64(s.p.prop.e)
    parts = []
    step = max(1, int(3e7 / ((case["d"] + 1) * case["width"] * case["hidden"])))
    with torch.set_grad_enabled(grad):
        for i in range(0, case["n"], step):
            lo, hi = (t64(a[i:i + step], grad) for a in (s.lo, s.hi))
            alpha = t64(s.alpha[i:i + step], grad) if s.alpha is not None else None
            row_lo, row_hi, slopes = _row_bounds64(W, b, C, e, lo, hi, alpha)
            if not grad:
                parts.append((row_lo, row_hi))
                continue
            ((row_lo * t64(s.g_lo[i:i + step])).sum() + (row_hi * t64(s.g_hi[i:i + step])).sum()).backward()
            d_alpha = alpha.grad if alpha is not None else torch.cat(
                [a.grad if a.grad is not None else torch.zeros_like(a) for a in slopes], dim=1)
            parts.append((row_lo.detach(), row_hi.detach(), d_alpha, lo.grad, hi.grad))
    whole = [torch.cat(p) for p in zip(*parts)]
    out = dict(zip(("row_lo", "row_hi", "d_alpha", "d_lo", "d_hi"), whole))
    if grad and case["weights"]:
        out["d_W"], out["d_b"] = [w.grad for w in W], [x.grad for x in b]
    return out
