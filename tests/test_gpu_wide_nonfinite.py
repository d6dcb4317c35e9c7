"""NaN and infinities through the wide adjoint (needs a GB300): a network of 40 inputs runs the general
products, the same network with inputs of no weight and no width added (64, 224 and 784 inputs) the
layer kernel's.  What is not finite in a box's gradients or bounds on the one is not finite on the
other, and the boxes beside it keep their bits."""
import numpy as np
import pytest

from workloads import generators as gen

from .gpu_common import random_sub_boxes

pytestmark = pytest.mark.gpu

D0, HIDDEN, R, N, BAD = 40, [48, 40, 33], 5, 6, 2
KEYS = ("row_lo", "row_hi", "d_alpha", "d_lo", "d_hi")


@pytest.fixture(scope="module")
def pkg():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2312_05890_gb300 as m
    return m


def _problem(scale=1.0):
    rng = np.random.default_rng(8)
    net = gen._mlp(rng, [D0] + HIDDEN + [6])
    for k in range(2):
        net.W[k] = (net.W[k] * np.float32(scale)).astype(np.float32)
    c = rng.random(D0)
    rows = [(rng.normal(size=6).astype(np.float32), float(rng.normal()), False) for _ in range(R)]
    return gen.Problem("nan", net, (c - 0.1).astype(np.float32), (c + 0.1).astype(np.float32), gen._prop([rows]), 3, 0)


def _pad(x, d):
    return np.concatenate([x, np.zeros(x.shape[:-1] + (d - D0,), np.float32)], axis=-1)


def _backward(pkg, p, d, lo, hi, g_lo, g_hi, alpha):
    with pkg.Counter(0) as c:
        c.load_network([_pad(p.net.W[0], d)] + list(p.net.W[1:]), p.net.b)
        c.set_box(_pad(p.lo, d), _pad(p.hi, d))
        c.set_property(p.prop.rows_per_clause, p.prop.C, p.prop.e, p.prop.strict)
        c.set_options(wide=1)
        r = c.margin_backward(_pad(lo, d), _pad(hi, d), g_lo, g_hi, alpha=alpha)
    return {k: r[k][:, :D0] if k in ("d_lo", "d_hi") else r[k] for k in KEYS}


def _inputs(p, seed):
    rng = np.random.default_rng(seed)
    lo, hi = random_sub_boxes(p, N, seed=seed)
    g_lo, g_hi = (rng.normal(size=(N, R)).astype(np.float32) for _ in range(2))
    return lo, hi, g_lo, g_hi, rng.uniform(0.05, 0.95, size=(N, sum(HIDDEN))).astype(np.float32)


@pytest.mark.parametrize("d", [64, 224, 784])
@pytest.mark.parametrize("free", [True, False])
@pytest.mark.parametrize("what", ["one nan", "all nan", "one inf", "all -inf", "sign bit nan"])
def test_gradients_of_a_diverged_loss(pkg, d, free, what):
    p = _problem()
    lo, hi, g_lo, g_hi, A = _inputs(p, d)
    A = A if free else None
    clean = _backward(pkg, p, d, lo, hi, g_lo, g_hi, A)
    assert all(np.isfinite(v).all() for v in clean.values())
    value = {"one nan": np.nan, "all nan": np.nan, "one inf": np.inf, "all -inf": -np.inf,
             "sign bit nan": np.array([0xFFFFFFFF], np.uint32).view(np.float32)[0]}[what]
    if what.startswith("all"):
        g_lo[BAD] = g_hi[BAD] = value
    else:
        g_hi[BAD, 1] = value
    want = _backward(pkg, p, D0, lo, hi, g_lo, g_hi, A)
    got = _backward(pkg, p, d, lo, hi, g_lo, g_hi, A)
    assert not np.isfinite(want["d_lo"][BAD]).any()
    others = np.arange(N) != BAD
    for k in KEYS:
        assert np.array_equal(np.isfinite(got[k]), np.isfinite(want[k])), k
        assert np.array_equal(got[k][others], clean[k][others]), k


@pytest.mark.parametrize("d", [64, 224, 784])
def test_a_forward_state_that_overflows(pkg, d):
    p = _problem(scale=1e20)              # the second layer's coefficients pass the largest float
    lo, hi, g_lo, g_hi, A = _inputs(p, 3)
    want = _backward(pkg, p, D0, lo, hi, g_lo, g_hi, A)
    got = _backward(pkg, p, d, lo, hi, g_lo, g_hi, A)
    assert not np.isfinite(want["row_hi"]).any() and not np.isfinite(want["row_lo"]).any()
    for k in ("row_lo", "row_hi"):
        assert not np.isfinite(got[k]).any(), k
    assert np.array_equal(np.isfinite(got["d_lo"]), np.isfinite(want["d_lo"]))


@pytest.mark.parametrize("d", [D0, 64, 224, 784])
def test_bounds_of_a_state_that_overflows_stay_sound(pkg, d):
    """The sound bounds drop a NaN coefficient; the row's N and E hold it, so no bound is finite."""
    p = _problem(scale=1e20)
    lo, hi = random_sub_boxes(p, N, seed=1)
    with pkg.Counter(0) as c:
        c.load_network([_pad(p.net.W[0], d)] + list(p.net.W[1:]), p.net.b)
        c.set_box(_pad(p.lo, d), _pad(p.hi, d))
        c.set_property(p.prop.rows_per_clause, p.prop.C, p.prop.e, p.prop.strict)
        c.set_options(wide=1)
        rl, rh, cls = c.bounds(_pad(lo, d), _pad(hi, d))
    assert not (rl > -np.inf).any() and not (rh < np.inf).any()
    assert (cls == 2).all()
