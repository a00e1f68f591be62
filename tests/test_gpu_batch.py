"""Batched stepping (qtt_step_many): independent PDFs of different grid, chi
and precision advanced together on their own streams give exactly the
states of stepping each alone."""
import pytest

import workload

pytestmark = pytest.mark.gpu
pkg = pytest.importorskip("paper_2407_09169_gb300")


@pytest.fixture(scope="module", autouse=True)
def lib(gpu_available):
    from paper_2407_09169_gb300 import build
    build.build()
    return pkg.load_library()


def _instances():
    return [
        workload.make_params({"bits": 3, "chi_max": 8}, seed=1, precision="fp32", omega=0.7, da=3.0),
        workload.make_params({"bits": 4, "chi_max": 16}, seed=2, precision="fp64"),
        workload.make_params({"bits": 4, "chi_max": 12}, seed=3, precision="bf16x3", da=0.2),
        workload.make_params({"bits": 3, "chi_max": 128}, seed=4, precision="fp64", exact=1, svd_rel_tol=0.0),
    ]


def test_step_many_matches_separate_steps():
    """The first steps run context by context (eager step, graph captures);
    from then on one parent graph per step embeds every context's step graph.
    Stepping one context alone in between changes the contexts' relative
    parities, so the parent graphs are rebuilt; every state stays bitwise
    equal to stepping the contexts one by one."""
    ps = _instances()
    batch = [pkg.qtt_init(p) for p in ps]
    alone = [pkg.qtt_init(p) for p in ps]
    try:
        pkg.qtt_step_many(batch, 6)
        batch[1].step(1)
        pkg.qtt_step_many(batch, 3)
        for i, c in enumerate(alone):
            c.step(10 if i == 1 else 9)
        for a, b in zip(batch, alone):
            assert a.scalars()["steps"] == b.scalars()["steps"]
            assert a.compare(b) == 0.0
    finally:
        for c in batch + alone:
            c.close()


def test_step_many_rejects_a_repeated_context():
    c = pkg.qtt_init(_instances()[0])
    try:
        with pytest.raises(pkg.QttError) as ei:
            pkg.qtt_step_many([c, c], 1)
        assert "twice" in str(ei.value)
    finally:
        c.close()


def test_sets_stepped_in_turn_match_separate_steps():
    """Five sets (more than are kept) stepped in turn, a context shared by two
    sets, and a set whose context is destroyed and made anew: every state stays
    bitwise that of stepping the contexts alone."""
    ps = _instances()[:2]
    sets = [[pkg.qtt_init(p) for p in ps] for _ in range(4)]
    alone = [pkg.qtt_init(p) for p in ps]
    fresh = None
    try:
        sets.append([sets[0][0], sets[1][1]])
        for _ in range(2):
            for s in sets:
                pkg.qtt_step_many(s, 4)
        sets[2][0].close()
        fresh = pkg.qtt_init(ps[0])
        sets[2][0] = fresh
        pkg.qtt_step_many(sets[2], 5)
        steps = {id(c): 8 for s in sets[:4] for c in s}
        steps[id(sets[0][0])] = steps[id(sets[1][1])] = 16
        steps[id(fresh)], steps[id(sets[2][1])] = 5, 13
        for j, a in enumerate(alone):
            done = 0
            for s in sorted(sets[:4], key=lambda s: steps[id(s[j])]):
                n = steps[id(s[j])]
                a.step(n - done)
                done = n
                assert s[j].scalars()["steps"] == n and s[j].compare(a) == 0.0
    finally:
        for c in {id(c): c for s in sets for c in s}.values():
            c.close()
        for c in alone:
            c.close()


def test_parent_graphs_go_with_their_contexts():
    """The parent graphs of a set are dropped when one of its contexts is
    destroyed, without another batch call, and no destroyed context stays
    noted; a set that does not hold it stays."""
    kept = lambda: pkg.qtt_selftest(14).tolist()
    ps = _instances()[:2]
    before = kept()[0]
    a, b = [pkg.qtt_init(p) for p in ps], [pkg.qtt_init(p) for p in ps]
    try:
        pkg.qtt_step_many(a, 4)
        pkg.qtt_step_many(b, 4)
        assert kept() == [before + 2, 0]
        a[0].close()
        assert kept() == [before + 1, 0]
        b[1].close()
        assert kept() == [before, 0]
        a[1].close()
        pkg.qtt_init(ps[0]).close()
        assert kept() == [before, 0]
    finally:
        for c in a + b:
            c.close()
