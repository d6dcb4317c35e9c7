"""Contexts of different networks in several host threads at once (needs a GB300): one context per
thread is what the header allows, so what a launch asks of a kernel (its shared memory among it)
must not depend on another thread's network."""
import threading

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


def _problem(d, hidden, R, seed):
    rng = np.random.default_rng(seed)
    net = gen._mlp(rng, [d] + hidden + [6])
    c = rng.random(d)
    rows = [(rng.normal(size=6).astype(np.float32), float(rng.normal()), False) for _ in range(R)]
    return gen.Problem("t", net, (c - 0.05).astype(np.float32), (c + 0.05).astype(np.float32), gen._prop([rows]), 3, seed)


KINDS = {   # networks that launch the same kernels with different amounts of shared memory
    "tile": [(6, [20, 20], 2), (6, [60, 60, 60], 4), (6, [40], 3), (6, [50] * 5, 2)],
    "wide": [(12, [300], 2), (12, [1000], 4), (12, [500, 500], 3), (12, [64], 4)],
    "layer": [(64, [300], 2), (784, [256], 4), (225, [1000, 130], 3), (200, [64, 64], 4)],
}


@pytest.mark.parametrize("kind", sorted(KINDS))
def test_contexts_in_threads(pkg, kind):
    probs = [_problem(*s, seed=i) for i, s in enumerate(KINDS[kind])]
    errors = []
    start = threading.Barrier(len(probs))

    def calls(c, p, lo, hi, g):
        a = c.bounds(lo, hi)
        r = c.margin_backward(lo, hi, g, -g)
        n = c.count(4)
        s = c.optimize_alpha(lo, hi, steps=1)
        return list(a) + [r[k] for k in sorted(r)] + list(s) + [n["unsafe_lo"], n["unsafe_hi"]]

    def work(p):
        try:
            lo, hi = random_sub_boxes(p, 9, seed=1)
            g = np.ones((9, p.prop.R), np.float32)
            with pkg.Counter(0) as c:
                c.set_problem(p)
                c.set_options(wide=0 if kind == "tile" else 1)
                first = calls(c, p, lo, hi, g)
                start.wait()
                for _ in range(100):
                    for a, b in zip(first, calls(c, p, lo, hi, g)):
                        assert np.array_equal(a, b)
        except BaseException as e:      # noqa: BLE001
            errors.append(repr(e))
            start.abort()
    th = [threading.Thread(target=work, args=(p,)) for p in probs]
    for t in th:
        t.start()
    for t in th:
        t.join()
    assert errors == []
