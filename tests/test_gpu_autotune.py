"""The autotuner keeps the resident form a context runs by default, on lattices
and schedules whose resident form is no candidate of form 1, and a shape once
set can be taken back (form 2)."""
import numpy as np
import pytest

from paper_1012_5082_gb300 import inputs as I

pytestmark = pytest.mark.gpu
COUNTERS = ("steps", "trials", "local_accepts", "global_accepts", "flips", "n_b")


@pytest.fixture(scope="module")
def V():
    from paper_1012_5082_gb300 import vcsgc
    return vcsgc


def _context(V, kind, cells, sched, alloy, R=2):
    lat = I.bcc_lattice(*cells)
    T, c0, phi = (1000.0, 0.5, 0.0) if alloy == "ising" else (900.0, 0.1, -2.2)
    types = np.concatenate([I.random_types(lat.n, int(c0 * lat.n), seed=r) for r in range(R)])
    return V.Context(lat, types, I.ising_tables() if alloy == "ising" else I.eam_tables(), phi, 0.02, T, c0=c0,
                     n_replicas=R, seed_r=np.arange(R, dtype=np.uint64) + np.uint64(9), sched=sched,
                     schedule={"sublattice": V.SCHED_SUBLATTICE, "blocks": V.SCHED_BLOCKS, "overlap": V.SCHED_OVERLAP}[kind])


CASES = [("blocks", (10, 10, 10), (5, 5, 5, 2, 2, 2), "eam"), ("blocks", (40, 40, 40), (5, 5, 5, 2, 2, 2), "ising"),
         ("overlap", (20, 30, 20), (10, 10, 10, 4, 4, 4), "eam"), ("sublattice", (48, 48, 48), (4, 4, 4), "ising")]


@pytest.mark.parametrize("steps", [5, 64])
@pytest.mark.parametrize("kind,cells,sched,alloy", CASES)
def test_autotune_keeps_the_resident_form(V, kind, cells, sched, alloy, steps):
    """These have no other resident candidate, and their per-step launches take
    two to four times as long."""
    g = _context(V, kind, cells, sched, alloy)
    assert g.cluster_sizes() == []
    block = g.autotune(steps)
    assert g.get_launch()[0] == 2 and g.get_launch()[1] == block in (64, 128, 256)
    ran = g.observables(0)["steps"]
    assert ran == 7 * (1 + steps)
    g.steps(90)
    h = _context(V, kind, cells, sched, alloy)
    h.set_launch(0, 128, 1)
    h.steps(ran + 90)
    for r in range(2):
        assert np.array_equal(g.types(r), h.types(r))
        og, oh = g.observables(r), h.observables(r)
        assert [og[k] for k in COUNTERS] == [oh[k] for k in COUNTERS] and og["flips"] > 0
    g.close()
    h.close()


def test_form_2_takes_a_shape_back(V):
    """Forms 0, 1, 2 in turn are one chain; a shape that a schedule change makes
    unusable is forgotten."""
    cells = (40, 40, 40)
    g, h = (_context(V, "sublattice", cells, (4, 4, 4), "eam") for _ in range(2))
    assert g.get_launch()[0] == 0
    for shape in ((0, 64, 0), (2, 256, 1), (1, 256, 4), (2, 64, 0)):
        g.set_launch(*shape)
        assert g.get_launch() == shape
        g.steps(20)
        g.steps(3)
    h.set_launch(0, 128, 1)
    h.steps(4 * 23)
    g.set_launch(1, 256, 4)
    for c in (g, h):
        c.set_schedule(V.SCHED_BLOCKS, (5, 5, 5, 2, 2, 2))
        c.steps(30)
    assert g.get_launch()[0] == 0
    for r in range(2):
        assert np.array_equal(g.types(r), h.types(r))
        og, oh = g.observables(r), h.observables(r)
        assert [og[k] for k in COUNTERS] == [oh[k] for k in COUNTERS] and og["flips"] > 0
    for bad in ((2, 512, 1), (2, 128, 2)):
        with pytest.raises(V.VcsgcError) as e:
            g.set_launch(*bad)
        assert e.value.code == -1
    g.close()
    h.close()


@pytest.mark.parametrize("shape", [None, (1, 256, 8)])
def test_profiled_steps_hold_no_allocation(V, shape):
    """The first profiled run of a length, whose draws need larger buffers than
    the calls before, takes what later ones take, not the allocation's time
    (which is more than the steps' own); and a context without a shape is
    profiled in the form its calls run."""
    g = _context(V, "sublattice", (80, 80, 80), (4, 4, 4), "eam", R=8)
    if shape:
        g.set_launch(*shape)
    for _ in range(3):
        g.steps(8)
    first = g.profile_steps(64)
    later = [g.profile_steps(64) for _ in range(5)]
    assert first[1] == 0.0 and all(q[1] == 0.0 for q in later)  # one launch of many steps: no commits
    assert first[0] < 1.6 * np.median([q[0] for q in later]), (first, later)
    g.close()


@pytest.mark.parametrize("kind,cells,sched,R", [
    ("blocks", (80, 80, 40), (20, 20, 20, 2, 2, 2), 2),   # a large lattice on few threads: pays from some 30 steps up
    ("sublattice", (8, 8, 8), (4, 4, 4), 200),            # two waves of CTAs: from about 10
    ("sublattice", (8, 8, 8), (4, 4, 4), 500),            # four: never
    ("sublattice", (24, 24, 24), (4, 4, 4), 700),         # five full ones: again
    ("blocks", (10, 10, 10), (5, 5, 5, 2, 2, 2), 5000),   # more CTAs than the GPU holds
])
def test_calls_of_any_length_are_one_chain(V, kind, cells, sched, R):
    """Lengths on both sides of the shortest call that runs resident, by size."""
    g, h = (_context(V, kind, cells, sched, "eam", R=R) for _ in range(2))
    h.set_launch(0, 128, 1)
    lengths = (8, 9, 11, 13, 20, 27, 31, 40, 64, 8)
    for n in lengths:
        g.steps(n)
    h.steps(sum(lengths))
    assert np.array_equal(g.types_all(), h.types_all())
    for og, oh in zip(g.observables_all(), h.observables_all()):
        assert [og[k] for k in COUNTERS] == [oh[k] for k in COUNTERS]
    g.close()
    h.close()


def test_the_form_follows_the_accepts(V):
    """One large lattice without the variance constraint, hot: every step is
    accepted and takes 5.6 us resident, 4.1 by the per-step launch, which the
    default form takes after its first calls.  One chain."""
    import time

    import torch
    lat = I.bcc_lattice(112, 112, 112)
    types = I.random_types(lat.n, lat.n // 3, seed=1)

    def chain(shape):
        g = V.Context(lat, types, I.eam_tables(), -2.1, 0.0, 5000.0, c0=0.3, seed=3)
        if shape:
            g.set_launch(*shape)
        us = []
        for _ in range(6):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            g.steps(1000)
            o = g.observables()
            us.append((time.perf_counter() - t0) * 1e3)
        out = g.types(), [o[k] for k in COUNTERS]
        g.close()
        return out, us

    (ta, oa), follows = chain(None)
    (tb, ob), resident = chain((1, 512, 16))
    assert np.array_equal(ta, tb) and oa == ob and oa[3] > 0.9 * oa[0]
    assert min(follows[2:]) < 0.85 * min(resident[2:]), (follows, resident)
