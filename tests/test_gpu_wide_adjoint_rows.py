"""The wide adjoint's row kernels with one and with four neurons a thread (needs a GB300): batches
large enough for four against the same boxes alone, which take one, bit for bit; layers at and
beside a warp's width and a block's 128 neurons."""
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


@pytest.mark.parametrize("d,hidden,n", [(128, [33, 32, 40], 65), (200, [130, 128], 66), (129, [127, 31, 257], 70),
                                        (784, [256, 256], 33)])
@pytest.mark.parametrize("free", [True, False])
def test_a_box_alone_and_in_a_batch(pkg, d, hidden, n, free):
    rng = np.random.default_rng(d + n)
    net = gen._mlp(rng, [d] + hidden + [6])
    c0 = rng.random(d)
    rows = [(rng.normal(size=6).astype(np.float32), float(rng.normal()), False) for _ in range(5)]
    p = gen.Problem("rows", net, (c0 - 0.02).astype(np.float32), (c0 + 0.02).astype(np.float32),
                    gen._prop([rows[:3], rows[3:]]), 3, 0)
    lo, hi = random_sub_boxes(p, n, seed=n)
    g_lo, g_hi = (rng.normal(size=(n, 5)).astype(np.float32) for _ in range(2))
    A = rng.uniform(0.0, 1.0, size=(n, sum(hidden))).astype(np.float32) if free else None
    with pkg.Counter(0) as c:
        c.set_problem(p)
        c.set_options(wide=1)
        whole = c.margin_backward(lo, hi, g_lo, g_hi, alpha=A)
        slopes = c.optimize_alpha(lo, hi, steps=3)
        for i in (0, 1, n // 2, n - 1):
            s = slice(i, i + 1)
            one = c.margin_backward(lo[s], hi[s], g_lo[s], g_hi[s], alpha=None if A is None else A[s])
            for k in one:
                assert np.array_equal(whole[k][s], one[k]), (k, i)
            for a, b in zip(slopes, c.optimize_alpha(lo[s], hi[s], steps=3)):
                assert np.array_equal(a[s], b), i
