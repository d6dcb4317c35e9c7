"""Networks loaded one after another into one context (needs a GB300): the kernels that lay out a
network's weights read what was uploaded for it, on the layer-kernel, wide, tensor-core and tile
paths, with the adjoint's transposed pieces and a gradient-split count's tables."""
import numpy as np
import pytest

from workloads import generators as gen

from .gpu_common import random_sub_boxes

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2312_05890_gb300 as m
    return m


def _problem(d, hidden, seed):
    rng = np.random.default_rng(seed)
    net = gen._mlp(rng, [d] + hidden + [6])
    c = rng.random(d)
    rows = [(rng.normal(size=6).astype(np.float32), float(rng.normal()), False) for _ in range(5)]
    return gen.Problem("net", net, (c - 0.05).astype(np.float32), (c + 0.05).astype(np.float32),
                       gen._prop([rows[:3], rows[3:]]), 3, seed)


def _answers(c, p, opt):
    lo, hi = random_sub_boxes(p, 3, seed=5)
    c.set_problem(p)
    out = list(c.bounds(lo, hi, want_err=True))
    if not opt.get("precision"):
        g = np.ones((3, 5), np.float32)
        r = c.margin_backward(lo, hi, g, -g)
        out += [r[k] for k in sorted(r)]
    return out


@pytest.mark.parametrize("d,hidden,opt", [(200, [1024, 1024, 1000], {}), (40, [700, 900], {}),
                                          (5, [50, 50, 50], dict(precision=1)), (9, [50, 50], {})])
def test_each_network_answers_as_in_a_fresh_context(pkg, d, hidden, opt):
    tile = {}
    if not opt and max(hidden) < 64:
        tile = dict(tile_boxes=8, tile_threads=256)   # (two contexts may time two tiles differently)
    with pkg.Counter(0) as kept:
        kept.set_options(**opt, **tile)
        for seed in range(6):
            p = _problem(d, hidden, seed)
            a = _answers(kept, p, opt)
            with pkg.Counter(0) as fresh:
                fresh.set_options(**opt, **tile)
                b = _answers(fresh, p, opt)
            for x, y in zip(a, b):
                assert np.array_equal(x, y), seed


def test_gradient_split_counts_of_two_problems(pkg):
    probs = [_problem(7, [30, 30], s) for s in (1, 2, 3)]

    def count(c, p):
        c.set_problem(p)
        r = c.count(8)
        return r["level_boxes"], r["unsafe_lo"], r["unsafe_hi"], c.split_set().tolist()
    with pkg.Counter(0) as kept:
        kept.set_options(split_rule=pkg.SPLIT_GRADIENT)
        for p in probs:
            a = count(kept, p)
            with pkg.Counter(0) as fresh:
                fresh.set_options(split_rule=pkg.SPLIT_GRADIENT)
                assert a == count(fresh, p)
