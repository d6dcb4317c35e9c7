"""Levels of few boxes (needs a GB300): the one-block compaction at its sizes' edges (runs of
1024 boxes, the last level it takes and the first it does not) and the smaller tiles that such
levels run, whole leaf sets against the FP64 oracle; the same counts allocation-free and resumed
across the change of compaction, re-checks included."""
import pytest

import oracle
from workloads import generators as gen

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2312_05890_gb300 as m
    return m


@pytest.mark.parametrize("name,D", [("tiny", 0), ("tiny", 1), ("acas", 10), ("acas", 12), ("acas", 13), ("nav", 11),
                                    ("rare", 14)])
def test_whole_leaf_sets(pkg, name, D):
    p = gen.make(name)
    want = oracle.count(p.net, p.lo, p.hi, p.prop, D)
    with pkg.Counter(0) as c:
        c.set_problem(p)
        c.set_options(record_leaves=1)
        got = c.count(D)
        codes, depth, cls = c.leaves()
        c.set_options()
        plain = c.count(D)
        lean = c.count_noalloc(D)
        cut = c.resume(c.checkpoint(D, D - 1)) if D > 0 else plain
    assert (got["unsafe_lo"], got["unsafe_hi"]) == (want.unsafe_lo, want.unsafe_hi)
    assert got["level_boxes"] == [lv["boxes"] for lv in want.levels]
    leaves = sorted(zip(codes.tolist(), depth.tolist(), cls.tolist()))
    assert len(leaves) == len(set(leaves)) and sum(1 << (D - t) for _, t, _ in leaves) == 1 << D
    for key in ("unsafe_lo", "unsafe_hi", "level_boxes", "level_safe", "level_unsafe", "level_undecided", "rechecked",
                "tie_leaves"):
        assert got[key] == plain[key] == lean[key] == cut[key], key


@pytest.mark.parametrize("D", [11, 12, 13, 14])
def test_full_levels(pkg, D):
    """Full levels of 2048 to 16384 boxes (hardly any navigation-shaped box is decided)."""
    p = gen.make("nav")
    want = oracle.count(p.net, p.lo, p.hi, p.prop, D)
    with pkg.Counter(0) as c:
        c.set_problem(p)
        got = c.count(D)
    assert got["level_boxes"] == [lv["boxes"] for lv in want.levels]
    assert (got["unsafe_lo"], got["unsafe_hi"]) == (want.unsafe_lo, want.unsafe_hi)
