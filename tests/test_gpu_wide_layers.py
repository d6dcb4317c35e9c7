"""The wide path's layer kernel at the edges of its tiles (needs a GB300): input counts at the
smallest it takes and around one and two column tiles, layer widths around one and two row
tiles and off the multiples of 8 and 32, one hidden layer (the property rows straight from the
first layer), 1 to 16 property rows, boxes beside a whole number of tiles; raw bounds against
the FP64 oracle, at the default and at supplied slopes, and in the other reading and activations."""
import numpy as np
import pytest

import oracle
from workloads import generators as gen

from .gpu_common import BOUND_RTOL, bound_errors, random_sub_boxes
from .test_gpu_alpha import _close, _split_alpha, _split_alpha_batch

pytestmark = pytest.mark.gpu

SHAPES = [  # d, hidden widths, property rows, boxes
    (63, [40, 24], 3, 5),        # the last input count of the general wide path
    (64, [8, 8], 1, 1),
    (65, [128, 129], 4, 3),
    (200, [33], 16, 7),
    (256, [31, 100, 17], 5, 2),
    (257, [130, 72], 9, 37),
    (513, [256, 257], 12, 4),
    (100, [60, 61, 62, 63], 13, 11),
    (784, [256, 256], 9, 160),
]


@pytest.fixture(scope="module")
def pkg():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2312_05890_gb300 as m
    return m


def _problem(d, hidden, R, act="relu"):
    rng = np.random.default_rng(d + sum(hidden))
    net = gen._mlp(rng, [d] + hidden + [6])
    net.act = [act] * len(hidden) if act != "relu" else []
    c = rng.random(d)
    lo, hi = (c - 0.01).astype(np.float32), (c + 0.01).astype(np.float32)
    rows = [(rng.normal(size=6).astype(np.float32), float(rng.normal()), False) for _ in range(R)]
    return gen.Problem("wide", net, lo, hi, gen._prop([rows]), 3, 0)


def _check(pkg, p, n, alpha=None, **opt):
    lo, hi = random_sub_boxes(p, n, seed=n)
    with pkg.Counter(0) as c:
        c.set_problem(p)
        c.set_options(wide=1, **opt)
        rl, rh, _, err = c.bounds(lo, hi, want_err=True, alpha=alpha)
        again = c.bounds(lo, hi, want_err=True, alpha=alpha)
    assert np.array_equal(rl, again[0]) and np.array_equal(rh, again[1])
    al = None if alpha is None else [a.astype(np.float64) for a in _split_alpha_batch(p.net, alpha)]
    olo, ohi = oracle.slr_forward(p.net, lo.astype(np.float64), hi.astype(np.float64), p.prop, alpha=al)[:2]
    scale = np.maximum(np.abs(olo), np.abs(ohi)) + (ohi - olo)
    assert np.all(rl <= olo + 1e-12 * scale) and np.all(rh >= ohi - 1e-12 * scale)
    return bound_errors(rl.astype(np.float64) + err, rh.astype(np.float64) - err, olo, ohi)


@pytest.mark.parametrize("d,hidden,R,n", SHAPES)
def test_raw_bounds(pkg, d, hidden, R, n):
    elo, ehi, _ = _check(pkg, _problem(d, hidden, R), n)
    assert elo.max() <= BOUND_RTOL and ehi.max() <= BOUND_RTOL, (elo.max(), ehi.max())


@pytest.mark.parametrize("d,hidden,R,n", SHAPES[1:6])
def test_raw_bounds_at_supplied_slopes(pkg, d, hidden, R, n):
    alpha = np.random.default_rng(d).random((n, sum(hidden)), dtype=np.float32)
    elo, ehi, _ = _check(pkg, _problem(d, hidden, R), n, alpha)
    assert elo.max() <= BOUND_RTOL and ehi.max() <= BOUND_RTOL, (elo.max(), ehi.max())


@pytest.mark.parametrize("act", ["tanh", "sigmoid"])
def test_widened_bounds_of_other_activations(pkg, act):
    # (the FP32 tanh/exp slopes carry about 2^-21; see the S-shaped tests' bar of 4e-5)
    elo, ehi, _ = _check(pkg, _problem(130, [40, 50], 3, act), 9)
    assert elo.max() <= 4e-5 and ehi.max() <= 4e-5, (elo.max(), ehi.max())


def test_more_boxes_than_a_chunk(pkg):
    """A second chunk of boxes reuses the state's buffers: the same bounds as alone."""
    p = _problem(784, [256, 256], 9)
    lo, hi = random_sub_boxes(p, 1400, seed=1)
    with pkg.Counter(0) as c:
        c.set_problem(p)
        rl, rh, _ = c.bounds(lo, hi)
        part = c.bounds(lo[1300:], hi[1300:])
    assert np.array_equal(rl[1300:], part[0]) and np.array_equal(rh[1300:], part[1])


@pytest.mark.parametrize("d,hidden,R,n", [(64, [8, 8], 1, 1), (223, [40], 3, 2), (224, [129, 33], 5, 3),
                                          (100, [60, 61, 62], 13, 4), (300, [256, 130], 9, 2)])
@pytest.mark.parametrize("free", [True, False])
def test_adjoint(pkg, d, hidden, R, n, free):
    """The adjoint's products on the same kernel (d + 1 columns), forward and through the
    transposed weights, against central differences at sampled coordinates."""
    p = _problem(d, hidden, R)
    rng = np.random.default_rng(d)
    lo, hi = random_sub_boxes(p, n, seed=n)
    H = sum(hidden)
    g_lo, g_hi = (rng.normal(size=(n, R)).astype(np.float32) for _ in range(2))
    A = rng.uniform(0.05, 0.95, size=(n, H)).astype(np.float32) if free else None
    a_idx = rng.choice(H, size=min(H, 30), replace=False)
    x_idx = rng.choice(d, size=20, replace=False)
    with pkg.Counter(0) as c:
        c.set_problem(p)
        c.set_options(wide=1)
        whole = c.margin_backward(lo, hi, g_lo, g_hi, alpha=A)
        for i in range(n):
            one = c.margin_backward(lo[i:i + 1], hi[i:i + 1], g_lo[i:i + 1], g_hi[i:i + 1],
                                    alpha=None if A is None else A[i:i + 1])
            for key in whole:
                assert np.array_equal(whole[key][i:i + 1], one[key]), key
    for i in (0, n - 1):
        fd = oracle.fd_gradients(p.net, lo[i], hi[i], p.prop,
                                 _split_alpha(p.net, A[i].astype(np.float64)) if free else None,
                                 g_hi[i].astype(np.float64), g_lo[i].astype(np.float64), h=1e-4, w_idx={},
                                 alpha_idx=a_idx if free else None, box_idx=x_idx)
        checks = [("d_lo", fd["lo"]), ("d_hi", fd["hi"])] + ([("d_alpha", np.concatenate(fd["alpha"]))] if free else [])
        for key, want in checks:
            ok, e = _close(whole[key][i], want, 2e-3)
            assert ok, (key, i, e)
