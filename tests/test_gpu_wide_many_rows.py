"""Properties of 13 to 16 rows behind layers so wide that the rows' weights pass 48 KB of shared
memory (needs a GB300): bounds, the adjoint and slope steps on the general wide path and on the
layer kernel, against the FP64 oracle."""
import numpy as np
import pytest

import oracle
from workloads import generators as gen

from .gpu_common import BOUND_RTOL, bound_errors, random_sub_boxes
from .test_gpu_alpha import _close

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2312_05890_gb300 as m
    return m


@pytest.mark.parametrize("d", [12, 64])
@pytest.mark.parametrize("width,R", [(768, 16), (769, 13), (1024, 12), (1024, 13), (1024, 16)])
def test_rows_beside_a_wide_last_layer(pkg, d, width, R):
    rng = np.random.default_rng(width + R + d)
    net = gen._mlp(rng, [d, width, 6])
    c0 = rng.random(d)
    rows = [(rng.normal(size=6).astype(np.float32), float(rng.normal()), False) for _ in range(R)]
    p = gen.Problem("rows", net, (c0 - 0.01).astype(np.float32), (c0 + 0.01).astype(np.float32), gen._prop([rows]), 3, 0)
    lo, hi = random_sub_boxes(p, 3, seed=2)
    g_lo, g_hi = (rng.normal(size=(3, R)).astype(np.float32) for _ in range(2))
    x_idx = rng.choice(d, size=6, replace=False)
    with pkg.Counter(0) as c:
        c.set_problem(p)
        c.set_options(wide=1)
        rl, rh, _, err = c.bounds(lo, hi, want_err=True)
        got = c.margin_backward(lo, hi, g_lo, g_hi)
        c.optimize_alpha(lo, hi, steps=2)
    olo, ohi = oracle.slr_forward(p.net, lo.astype(np.float64), hi.astype(np.float64), p.prop)[:2]
    assert np.all(rl <= olo) and np.all(rh >= ohi)
    elo, ehi, _ = bound_errors(rl.astype(np.float64) + err, rh.astype(np.float64) - err, olo, ohi)
    assert elo.max() <= BOUND_RTOL and ehi.max() <= BOUND_RTOL
    fd = oracle.fd_gradients(p.net, lo[0], hi[0], p.prop, None, g_hi[0].astype(np.float64), g_lo[0].astype(np.float64),
                             h=1e-4, w_idx={}, alpha_idx=None, box_idx=x_idx)
    for key, want in (("d_lo", fd["lo"]), ("d_hi", fd["hi"])):
        ok, e = _close(got[key][0], want, 2e-3)
        assert ok, (key, e)
