"""The adjoint over the edges of its warp-per-box form (needs a GB300): input counts at
the column paddings (1, 3 | 4, 5 | 6, 7 | 8 the block form), widths at one, two and four
rows a lane, against FP64 central differences of the oracle; and batches that end inside
a block against the same boxes one at a time."""
import numpy as np
import pytest

import oracle
from workloads import generators as gen

from .gpu_common import random_sub_boxes
from .test_gpu_alpha import _close, _split_alpha

pytestmark = pytest.mark.gpu

# (d, hidden widths, outputs); the first of each pair of neighbours is the last of its form
SHAPES = [(1, [1], 1), (3, [32], 2), (4, [33, 32], 3), (5, [64, 64], 5), (6, [65, 31], 2), (7, [128, 17], 4),
          (7, [129], 3), (8, [40, 24], 3), (5, [128, 128], 4), (2, [7, 6, 5, 4], 2)]


@pytest.fixture(scope="module")
def pkg():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2312_05890_gb300 as m
    return m


def _problem(d, hidden, out, seed):
    rng = np.random.default_rng(seed)
    net = gen._mlp(rng, [d] + hidden + [out])
    lo = rng.uniform(-0.5, 0.0, size=d).astype(np.float32)
    hi = (lo + rng.uniform(0.1, 0.4, size=d)).astype(np.float32)
    rows = [(rng.normal(size=out).astype(np.float32), float(rng.normal()), False) for _ in range(3)]
    return gen.Problem("shape", net, lo, hi, gen._prop([rows[:2], rows[2:]]), 4, seed)


@pytest.mark.parametrize("d,hidden,out", SHAPES)
@pytest.mark.parametrize("free", [True, False])
def test_adjoint_over_shapes(pkg, d, hidden, out, free):
    p = _problem(d, hidden, out, 7 * d + sum(hidden))
    rng = np.random.default_rng(d + out)
    H, n = sum(hidden), 19
    lo, hi = random_sub_boxes(p, n, seed=3)
    g_lo, g_hi = (rng.normal(size=(n, 3)).astype(np.float32) for _ in range(2))
    A = rng.uniform(0.05, 0.95, size=(n, H)).astype(np.float32) if free else None
    w_idx = {k: rng.choice(w.size, size=min(w.size, 12), replace=False) for k, w in enumerate(p.net.W)}
    a_idx = rng.choice(H, size=min(H, 40), replace=False)
    with pkg.Counter(0) as c:
        c.set_problem(p)

        def grads(s):
            return c.margin_backward(lo[s], hi[s], g_lo[s], g_hi[s], alpha=A[s] if free else None, weights=True)
        whole = grads(slice(0, n))
        single = [grads(slice(i, i + 1)) for i in range(n)]
        plain = c.margin_backward(lo, hi, g_lo, g_hi, alpha=A)
    # the same sums per box, however the boxes share blocks; weight gradients add up
    for key in ("row_lo", "row_hi", "d_alpha", "d_lo", "d_hi"):
        assert np.array_equal(whole[key], np.concatenate([s[key] for s in single])), key
        assert np.array_equal(whole[key], plain[key]), key
    for key in ("d_W", "d_b"):
        for k in range(len(p.net.W)):
            parts = np.stack([s[key][k] for s in single]).astype(np.float64)
            # float32 sums of the boxes' terms: 2^-24 per addition on the sum of magnitudes,
            # doubled for the two dot products inside a term (2 (d + 1) additions each)
            tol = 2.0 * (n + 2 * (d + 1) + 8) * 2.0 ** -24 * np.abs(parts).sum(0).max() + 1e-30
            assert np.abs(whole[key][k] - parts.sum(0)).max() <= tol, (key, k)
    for i in (0, n - 1):
        fd = oracle.fd_gradients(p.net, lo[i], hi[i], p.prop,
                                 _split_alpha(p.net, A[i].astype(np.float64)) if free else None,
                                 g_hi[i].astype(np.float64), g_lo[i].astype(np.float64), w_idx=w_idx,
                                 alpha_idx=a_idx if free else None)
        checks = [("d_lo", single[i]["d_lo"][0], fd["lo"]), ("d_hi", single[i]["d_hi"][0], fd["hi"])]
        if free:
            checks.append(("d_alpha", single[i]["d_alpha"][0], np.concatenate(fd["alpha"])))
        for k in range(len(p.net.W)):
            checks.append((f"d_W{k}", single[i]["d_W"][k], fd["W"][k]))
            checks.append((f"d_b{k}", single[i]["d_b"][k], fd["b"][k]))
        for key, got, want in checks:
            ok, e = _close(got, want, 2e-3)
            assert ok, (key, i, e)


@pytest.mark.parametrize("per_sm", [0, 1, 16, 20, 28])
@pytest.mark.parametrize("weights", [False, True])
def test_adjoint_rounds(pkg, per_sm, weights):
    """Around a full round of one block per SM: every box is taken once, in whatever slot."""
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    p = _problem(5, [40, 33], 4, 11)
    rng = np.random.default_rng(per_sm)
    with pkg.Counter(0) as c:
        c.set_problem(p)
        for n in (per_sm * sms + 1, max(per_sm, 1) * sms, max(per_sm, 1) * sms - 1):
            lo, hi = random_sub_boxes(p, n, seed=n)
            g_lo, g_hi = (rng.normal(size=(n, 3)).astype(np.float32) for _ in range(2))
            a = c.margin_backward(lo, hi, g_lo, g_hi, weights=weights)
            b = c.margin_backward(lo[::-1], hi[::-1], g_lo[::-1], g_hi[::-1], weights=weights)
            for key in ("row_lo", "row_hi", "d_lo", "d_hi"):
                assert np.array_equal(a[key], b[key][::-1]), (key, n)
            if weights:
                same = [np.repeat(x[:1], n, axis=0) for x in (lo, hi, g_lo, g_hi)]
                one = c.margin_backward(*[x[:1] for x in same], weights=True)
                many = c.margin_backward(*same, weights=True)
                for key in ("d_W", "d_b"):
                    for k in range(len(p.net.W)):
                        want = n * one[key][k].astype(np.float64)
                        # as above: n equal terms, 2 (d + 1) additions inside each
                        tol = 2.0 * (n + 2 * 6 + 8) * 2.0 ** -24 * np.abs(want).max() + 1e-30
                        assert np.abs(many[key][k] - want).max() <= tol, (key, k, n)
