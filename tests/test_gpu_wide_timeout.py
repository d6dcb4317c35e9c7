"""Every entry point that runs the wide path's bounded waits reports one that gave up (needs a GB300).
The wait is the self-check's, on a barrier that nothing completes, run among the call's own kernels;
the call returns SLR_ETIMEOUT and the same call afterwards gives the same answer as before."""
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


def _problem(d):
    rng = np.random.default_rng(d)
    net = gen._mlp(rng, [d, 40, 30, 6])
    c = rng.random(d)
    rows = [(rng.normal(size=6).astype(np.float32), float(rng.normal()), False) for _ in range(4)]
    return gen.Problem("wait", net, (c - 0.05).astype(np.float32), (c + 0.05).astype(np.float32),
                       gen._prop([rows[:2], rows[2:]]), 4, 0)


@pytest.mark.parametrize("d", [40, 64])      # the general products, the layer kernel
@pytest.mark.parametrize("call", ["bounds", "backward", "optimise", "count", "count with slopes", "gradient split"])
def test_a_wait_that_gives_up_is_reported(pkg, d, call):
    p = _problem(d)
    lo, hi = random_sub_boxes(p, 7, seed=1)
    g = np.ones((7, 4), np.float32)
    with pkg.Counter(0) as c:
        c.set_problem(p)
        c.set_options(wide=1, alpha_steps=2 if call == "count with slopes" else 0,
                      split_rule=1 if call == "gradient split" else 0)

        def run():
            if call == "bounds":
                return list(c.bounds(lo, hi))
            if call == "backward":
                r = c.margin_backward(lo, hi, g, -g)
                return [r[k] for k in sorted(r)]
            if call == "optimise":
                r = c.optimize_alpha(lo, hi, steps=3)
                return [r[k] for k in sorted(r)] if isinstance(r, dict) else list(r)
            r = c.count(4)
            return [r["level_boxes"], r["unsafe_lo"], r["unsafe_hi"]]
        before = run()
        assert pkg.load_library().slr_internal_wait_on_next(c.ctx, 4096) == 0
        with pytest.raises(pkg.SlrError, match="ETIMEOUT"):
            run()
        after = run()
    for a, b in zip(before, after):
        assert np.array_equal(a, b)
