"""The adjoint's warp-per-box form against its block form, bit for bit (needs a GB300): a network of
at most 7 inputs runs the first, the same network with inputs of no weight and no width added (8 in
all) the second.  Such an input adds exact zeros to every sum."""
import numpy as np
import pytest

from workloads import generators as gen

from .gpu_common import random_sub_boxes

pytestmark = pytest.mark.gpu

SHAPES = [(1, [1]), (2, [32]), (3, [33, 20]), (4, [64, 64, 7]), (5, [50] * 6), (6, [65, 31]), (7, [128, 17])]


@pytest.fixture(scope="module")
def pkg():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2312_05890_gb300 as m
    return m


def _pad(x):
    return np.concatenate([x, np.zeros(x.shape[:-1] + (8 - x.shape[-1],), np.float32)], axis=-1)


@pytest.mark.parametrize("d,hidden", SHAPES)
@pytest.mark.parametrize("upstream", ["random", "one nan", "one inf"])
def test_both_forms(pkg, d, hidden, upstream):
    rng = np.random.default_rng(d)
    net = gen._mlp(rng, [d] + hidden + [4])
    lo0 = rng.uniform(-0.5, 0.0, size=d).astype(np.float32)
    hi0 = (lo0 + rng.uniform(0.1, 0.5, size=d)).astype(np.float32)
    rows = [(rng.normal(size=4).astype(np.float32), float(rng.normal()), False) for _ in range(3)]
    p = gen.Problem("form", net, lo0, hi0, gen._prop([rows[:2], rows[2:]]), 3, 0)
    n = 41
    lo, hi = random_sub_boxes(p, n, seed=d)
    g_lo, g_hi = (rng.normal(size=(n, 3)).astype(np.float32) for _ in range(2))
    if upstream != "random":
        g_lo[7, 1] = np.nan if upstream == "one nan" else np.inf
    A = rng.uniform(-0.1, 1.1, size=(n, sum(hidden))).astype(np.float32)
    out = []
    for W0, box, b in ((net.W[0], (p.lo, p.hi), (lo, hi)),
                       (_pad(net.W[0]), (_pad(p.lo), _pad(p.hi)), (_pad(lo), _pad(hi)))):
        with pkg.Counter(0) as c:
            c.load_network([W0] + list(net.W[1:]), net.b)
            c.set_box(*box)
            c.set_property(p.prop.rows_per_clause, p.prop.C, p.prop.e, p.prop.strict)
            r = []
            for alpha in (A, None):
                m = c.margin_backward(*b, g_lo, g_hi, alpha=alpha)
                r += [m["row_lo"], m["row_hi"], m["d_alpha"], m["d_lo"][:, :d], m["d_hi"][:, :d]]
            r.append(c.optimize_alpha(*b, steps=4)[3])
            out.append(r)
    for i, (x, y) in enumerate(zip(*out)):
        assert np.array_equal(x, y, equal_nan=True), i
