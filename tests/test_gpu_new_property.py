"""A new property for the network already on the device (needs a GB300): counts, bounds, the
adjoint and the re-check after a change of rows, clauses, strictness or their number equal those
of a fresh context, on the tile, tensor-core, wide and layer-kernel paths."""
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


def _image():
    rng = np.random.default_rng(4)
    net = gen._mlp(rng, [90, 40, 33, 6])
    c = rng.random(90)
    p = gen.Problem("image", net, (c - 0.02).astype(np.float32), (c + 0.02).astype(np.float32), None, 6, 0)
    p.prop = gen._prop([[(gen._unit(6, j) - gen._unit(6, 0), 0.0, False)] for j in range(1, 6)])
    return p


def _properties(n_out, rows):
    """Properties of `rows` rows, then one of another number, then the first again."""
    rng = np.random.default_rng(n_out)

    def some(m, strict, per_clause):
        r = [(rng.normal(size=n_out).astype(np.float32), float(rng.normal(0, 0.3)), strict) for _ in range(m)]
        return gen._prop([r[i:i + per_clause] for i in range(0, m, per_clause)])
    first = some(rows, True, 1)
    return [first, some(rows, False, 2), some(rows, True, rows), some(rows + 1, False, 1), first]


@pytest.mark.parametrize("name,opt,D", [("tiny", {}, 10), ("acas", {}, 9), ("acas", dict(precision=1), 8),
                                        ("acas", dict(wide=1), 8), ("image", {}, 5), ("acas", dict(relax_mode=1), 9),
                                        ("acas", dict(fp64_recheck=0), 9)])
def test_same_as_a_fresh_context(pkg, name, opt, D):
    p = _image() if name == "image" else gen.make(name)
    lo, hi = random_sub_boxes(p, 23, seed=2)
    keys = ("unsafe_lo", "unsafe_hi", "level_boxes", "level_safe", "level_unsafe", "tie_leaves")
    with pkg.Counter(0) as kept:
        kept.load_network(p.net.W, p.net.b)
        kept.set_box(p.lo, p.hi)
        kept.set_options(**opt)
        for prop in _properties(p.net.W[-1].shape[0], p.prop.R):
            g = np.ones((23, prop.R), np.float32)

            def answers(c):
                out = [c.count(D)]
                rows = c.bounds(lo, hi, want_err=True)
                grads = c.margin_backward(lo, hi, g, -g) if not opt.get("relax_mode") else {}
                return out[0], rows, grads
            kept.set_property(prop.rows_per_clause, prop.C, prop.e, prop.strict)
            a = answers(kept)
            with pkg.Counter(0) as fresh:
                fresh.load_network(p.net.W, p.net.b)
                fresh.set_box(p.lo, p.hi)
                tile = {} if a[0]["tile"][1] == 0 else dict(tile_boxes=a[0]["tile"][0], tile_threads=a[0]["tile"][1])
                fresh.set_options(**opt, **tile)
                fresh.set_property(prop.rows_per_clause, prop.C, prop.e, prop.strict)
                b = answers(fresh)
            assert {k: a[0][k] for k in keys} == {k: b[0][k] for k in keys}
            for x, y in zip(a[1], b[1]):
                assert np.array_equal(x, y)
            for k in a[2]:
                assert np.array_equal(a[2][k], b[2][k]), k
