"""Kernel launches of a count (needs a GB300): each level takes the same number whatever the form of
its FP64 re-check (both stages of the default one run in one launch)."""
import pytest

from workloads import generators as gen

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2312_05890_gb300 as m
    return m


@pytest.mark.parametrize("name,D", [("acas", 15), ("tiny", 13)])
def test_every_recheck_is_one_launch_a_level(pkg, name, D):
    launches = {}
    with pkg.Counter(0) as c:
        c.set_problem(gen.make(name))
        for form in (dict(recheck_pairs=1), dict(recheck_pairs=0), dict(recheck_cluster=1), dict(fp64_recheck=0)):
            c.set_options(**form)
            launches[tuple(form.items())] = c.count(D)["launches"]
    a, b, cluster, none = launches.values()
    assert a == b == cluster == none + D + 1
