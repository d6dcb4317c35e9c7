"""The FP32 tile of a call (needs a GB300).  A tile decides the last bits of a bound (the order of
its sums, and the box its constants are relative to), so a tile that the caller sets runs every
call, of few boxes too, and a batched problem runs the tile its result names at every step,
whatever it is batched with."""
import copy

import numpy as np
import pytest

from workloads import generators as gen

from .gpu_common import random_sub_boxes

pytestmark = pytest.mark.gpu

KEYS = ("unsafe_lo", "unsafe_hi", "level_boxes", "level_safe", "level_unsafe", "level_undecided")


@pytest.fixture(scope="module")
def pkg():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2312_05890_gb300 as m
    return m


@pytest.mark.parametrize("T,NT", [(20, 256), (16, 256), (8, 256), (4, 128)])
def test_a_set_tile_runs_calls_of_few_boxes(pkg, T, NT):
    """The first whole tiles of a large call are the tiles of a small one: the same bits."""
    p = gen.make("acas")
    lo, hi = random_sub_boxes(p, 20000, seed=3)
    with pkg.Counter(0) as c:
        c.set_problem(p)
        c.set_options(tile_boxes=T, tile_threads=NT)
        many = c.bounds(lo, hi, want_err=True)
        best = c.optimize_alpha(lo[:4096], hi[:4096], steps=2)
        for n in (T, 3 * T, 40 * T):
            few = c.bounds(lo[:n], hi[:n], want_err=True)
            for a, b in zip(many, few):
                assert np.array_equal(a[:n], b), n
            slopes = c.optimize_alpha(lo[:n], hi[:n], steps=2)
            for a, b in zip(best, slopes):
                assert np.array_equal(a[:n], b), n


def _shifted(p, e):
    q = copy.deepcopy(p)
    q.prop = gen._prop([[(p.prop.C[0], float(e), False)]])
    return q


def _threshold(pkg, p, **opt):
    """The largest float e with which the root box is SAFE (y + e < 0 everywhere) at a tile."""
    with pkg.Counter(0) as c:
        c.set_problem(_shifted(p, 0.0))
        c.set_options(fp64_recheck=0, **opt)

        def safe(e):
            c.set_property(np.array([1], np.int32), p.prop.C[:1], np.array([e], np.float32), np.zeros(1, np.uint8))
            return c.count(0)["level_safe"][0] == 1
        a, b = np.float32(-1e6), np.float32(1e6)
        assert safe(a) and not safe(b)
        while True:
            m = np.float32((np.float64(a) + np.float64(b)) / 2)
            if m == a or m == b:
                return a
            if safe(m):
                a = m
            else:
                b = m


def _separated(pkg):
    """A problem and an e between the thresholds of the batch's tile and of the 4-box tile."""
    for seed in range(12):
        p = gen.acas_shaped(seed)
        with pkg.Counter(0) as c:
            c.set_options(fp64_recheck=0)
            T = c.count_batch([_shifted(p, 0.0)], [0])[0]["tile"][0]
        at = {t: _threshold(pkg, p, tile_boxes=t, tile_threads=256) for t in (T, 4)}
        if at[T] != at[4]:
            return _shifted(p, max(at.values())), T
    pytest.fail("the tile set by the caller does not change any bit of the root box's bounds")


def test_a_batched_problem_does_not_depend_on_the_others(pkg):
    q, T = _separated(pkg)
    with pkg.Counter(0) as c:
        c.set_problem(q)
        c.set_options(fp64_recheck=0, tile_boxes=T, tile_threads=256)
        want = c.count(0)
        c.set_options(fp64_recheck=0, tile_boxes=4, tile_threads=256)
        assert c.count(0)["level_safe"] != want["level_safe"]
        for n in (1, 3, 700):
            got = c.count_batch([q] * n, [0] * n)
            for r in (got[0], got[-1]):
                assert r["tile"][0] == T
                assert {k: r[k] for k in KEYS} == {k: want[k] for k in KEYS}, n


@pytest.mark.parametrize("name,D", [("acas", 9), ("tiny", 13), ("nav", 8)])
def test_batched_counts_without_the_recheck(pkg, name, D):
    """Without the FP64 re-check a problem's classes are the FP32 tile's own: batched with others,
    or alone, they are the single count's on the tile that the batch names."""
    p = gen.make(name)
    others = [gen.tiny(1), gen.acas_shaped(3), gen.rare_violation(0)]
    with pkg.Counter(0) as c:
        c.set_options(fp64_recheck=0)
        alone = c.count_batch([p], [D])[0]
        mixed = c.count_batch(others + [p], [6, 7, 8, D])[3]
        many = c.count_batch([p] * 30, [D] * 30)[11]
        c.set_problem(p)
        for r in (alone, mixed, many):
            c.set_options(fp64_recheck=0, tile_boxes=r["tile"][0], tile_threads=256)
            want = c.count(D)
            for k in KEYS:
                assert r[k] == want[k], k


def test_checkpoints_keep_the_tiles_of_their_count(pkg):
    """A checkpoint of a count on tiles of the library's choosing resumes on them in a context with
    a tile of its own, one of a set tile on that tile; a version-3 state (no word on this) as the
    library's choice."""
    p = gen.make("acas")
    D, t = 13, 5
    with pkg.Counter(0) as c, pkg.Counter(0) as other:
        c.set_problem(p)
        free = c.count(D)
        state = c.checkpoint(D, t)
        other.set_problem(p)
        other.set_options(tile_boxes=4, tile_threads=128)
        keys = KEYS + ("rechecked", "rechecked_fp64", "tie_leaves", "tile")
        assert {k: other.resume(state)[k] for k in keys} == {k: free[k] for k in keys}
        own = other.count(D)
        assert {k: c.resume(other.checkpoint(D, t))[k] for k in keys} == {k: own[k] for k in keys}
        assert tuple(c.count(D)["tile"]) == tuple(free["tile"])
        head = 48                                   # a version-3 header: up to the tile
        old = state[:4] + (3).to_bytes(4, "little") + state[8:head] + state[head + 8:]
        assert {k: other.resume(old)[k] for k in keys} == {k: free[k] for k in keys}
