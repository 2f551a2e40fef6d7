"""Colour steps with species-dependent densities from the float entries and the
embedding cubics (csrc/kernels_multi.cu: k_multi_propose<2> and <3> without the
table, the float branch of the commit): what two species use where the
re-embedding table has no memory, and more than two where no fixed-point format
fits their tables.  Small uneven lattices, one period per axis, periods other
than four, several replicas, against the oracle a stretch at a time."""
import math

import numpy as np
import pytest

import oracle as O
from oracle import mlp as M
from paper_1012_5082_gb300 import inputs as I

pytestmark = pytest.mark.gpu
A = 2.855
SHELL_R = np.array([A * math.sqrt(3) / 2, A, A * math.sqrt(2), A * math.sqrt(11) / 2, A * math.sqrt(3)])
SHELL_N = np.array([8, 6, 12, 24, 8])
CELLS = [((4, 4, 4), (4, 4, 4), 2), ((8, 4, 12), (4, 4, 4), 3), ((10, 5, 15), (5, 5, 5), 1), ((12, 8, 10), (6, 4, 5), 1),
         ((16, 12, 20), (4, 4, 4), 2)]


@pytest.fixture(scope="module")
def V():
    from paper_1012_5082_gb300 import vcsgc
    return vcsgc


def _agree(g, orcs, ties=0):
    for r, o in enumerate(orcs):
        og, oo = g.observables(r), o.obs()
        assert oo["near_ties"] == og["near_ties"] == ties
        assert np.array_equal(g.types(r), o.types), r
        for k in ("trials", "local_accepts", "global_trials", "global_accepts", "flips", "steps"):
            assert og[k] == oo[k], (r, k, og[k], oo[k])
        # energies of both are sums from scratch (the GPU's) or of steps (the oracle's)
        assert abs(og["energy"] - oo["energy"]) <= 1e-9 * abs(oo["energy"])


@pytest.mark.parametrize("cells,period,R", CELLS)
def test_two_species_between_table_and_cubics(V, cells, period, R):
    """The form changes between stretches: one chain, and counts kept or rebuilt."""
    tab = I.eam_tables(I.multi_eam_params(2, dens_scale=(1.0, 1.25)))
    lat = I.bcc_lattice(*cells)
    kappa, T, c0, phi = 0.02, 1200.0, 0.1, [-2.2]
    types = np.stack([I.multi_random_types(lat.n, [lat.n // 10], seed=r + 3) for r in range(R)])
    seeds = np.arange(R, dtype=np.uint64) + np.uint64(lat.n)
    g = V.Multi(lat, types, tab, phi, kappa, T, c0=c0, seed_r=seeds, period=period)
    orcs = []
    for r in range(R):
        o = O.MultiSystem(lat, types[r], tab)
        o.set_params(phi, [kappa], T, c0=[c0], seed=int(seeds[r]))
        o.schedule_sublattice(cells, period)
        orcs.append(o)
    for table, n in ((0, 1), (0, 70), (1, 5), (0, 6), (0, 1), (1, 66), (0, 64)):
        g.set_table(table)
        g.steps(n)
        for o in orcs:
            o.parallel_steps(n)
        _agree(g, orcs)
        if n == 6:
            g.set_types(orcs[0].types, 0)  # the entries of one replica written again
    assert sum(g.observables(r)["flips"] for r in range(R)) > 0
    g.close()


@pytest.mark.parametrize("cells,period,R", CELLS[1:])
def test_delayed_acceptance_from_the_cubics(V, cells, period, R):
    """A network that predicts a constant: the two-stage chain, also across a
    change of form, which takes the counts over."""
    tab = I.eam_tables(I.multi_eam_params(2, dens_scale=(1.0, 1.25)))
    lat = I.bcc_lattice(*cells)
    kappa, T, c0, phi = 0.02, 1200.0, 0.1, -2.2
    types = I.random_types(lat.n, lat.n // 10, seed=5)
    orcs = []
    for r in range(R):
        o = O.System(lat, types, tab)
        o.set_params(phi, kappa, T, c0=c0, seed=50 + r)
        o.schedule_sublattice(cells, period)
        o.set_shells(SHELL_R)
        orcs.append(o)
    p = np.zeros(M.NPARAM, np.float32)
    p[-1] = np.float32(np.mean([orcs[0].delta_e(i) for i in np.nonzero(types == 0)[0][:300]]))
    s = V.Surrogate(p)
    g = V.Multi(lat, np.tile(types, (R, 1)), tab, [phi], kappa, T, c0=c0, seed_r=np.arange(50, 50 + R, dtype=np.uint64),
                period=period)
    g.set_surrogate(s)
    for o in orcs:
        o.set_surrogate("mlp", p.astype(np.float64))
    for table, n in ((0, 3), (0, 130), (1, 64), (0, 67)):
        g.set_table(table)
        g.steps(n)
        for o in orcs:
            o.parallel_steps(n)
        for r, o in enumerate(orcs):
            og, oo = g.observables(r), o.obs()
            assert oo["near_ties"] == og["near_ties"] == 0
            assert np.array_equal(g.types(r), o.types)
            for k in ("trials", "local_accepts", "global_accepts", "flips", "stage1_accepts"):
                assert og[k] == oo[k], (r, k)
    assert g.observables(0)["flips"] > 0
    X, _ = g.features()
    X = X.cpu().numpy()
    for i in range(0, lat.n, 7):
        assert np.array_equal(X[i], orcs[0].descriptor(i))
    s.close()
    g.close()


@pytest.mark.parametrize("K,ds,phi", [(3, (1.0, 0.02, 0.5), [-2.0, -2.0]), (4, (1.0, 0.02, 0.5, 1.2), [-2.0, -2.0, -2.0])])
@pytest.mark.parametrize("cells,period,R", CELLS)
def test_more_species_without_a_fixed_point_format(V, K, ds, phi, cells, period, R):
    """A species of next to no density: a shell's difference exceeds the smallest
    screened argument, so that an entry of 0 could reach the range."""
    p = I.multi_eam_params(K, dens_scale=ds)
    Fd = np.array([[p.dens(t, r)[0] for t in range(K)] for r in SHELL_R])
    dmax = max(np.ptp(f) for f in Fd)
    lowest = (SHELL_N * Fd.min(1)).sum() - dmax
    tab = I.eam_tables(p)
    assert dmax > max(lowest, tab.drho)
    lat = I.bcc_lattice(*cells)
    kappa, T, c0 = 0.02, 2500.0, 0.1
    types = np.stack([I.multi_random_types(lat.n, [lat.n // 10] * (K - 1), seed=r + 3) for r in range(R)])
    seeds = np.arange(R, dtype=np.uint64) + np.uint64(lat.n)
    g = V.Multi(lat, types, tab, phi, kappa, T, c0=c0, seed_r=seeds, period=period)
    with pytest.raises(V.VcsgcError) as e:
        g.set_table(1)
    assert e.value.code == -8
    orcs = []
    for r in range(R):
        o = O.MultiSystem(lat, types[r], tab)
        o.set_params(phi, [kappa] * (K - 1), T, c0=[c0] * (K - 1), seed=int(seeds[r]))
        o.schedule_sublattice(cells, period)
        orcs.append(o)
    for n in (1, 1, 6, 64, 70):
        g.steps(n)
        for o in orcs:
            o.parallel_steps(n)
        _agree(g, orcs)
    assert sum(g.observables(r)["flips"] for r in range(R)) > 0
    g.close()


def test_the_form_follows_the_flips(V):
    """A hot chain flips tens of thousands of sites a step and runs from the cubics
    after its first calls.  It is the chain of the table alone, and the time per
    step says which form ran: hot, 64^3 x 8 takes 119 us with the table and 65
    from the cubics."""
    import time

    import torch
    tab = I.eam_tables(I.multi_eam_params(2, dens_scale=(1.0, 1.25)))
    lat = I.bcc_lattice(64, 64, 64)
    R = 8
    types = np.stack([I.multi_random_types(lat.n, [lat.n // 3], seed=r) for r in range(R)])

    def chain(table):
        g = V.Multi(lat, types, tab, [-1.5], 0.0, 20000.0, c0=0.3, seed_r=np.arange(R, dtype=np.uint64))
        if table is not None:
            g.set_table(table)
        us = []
        for _ in range(6):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            g.steps(256)
            o = g.observables(0)
            us.append((time.perf_counter() - t0) / 256 * 1e6)
        out = [g.types(r) for r in range(R)], o["flips"], o["local_accepts"]
        g.close()
        return out, us

    (ta, fa, la), hot = chain(None)
    (tb, fb, lb), fixed = chain(1)
    assert fa == fb > 256 * 6 * 1000 and la == lb and all(np.array_equal(x, y) for x, y in zip(ta, tb))
    assert min(hot[2:]) < 0.75 * min(fixed[2:]), (hot, fixed)


def test_captured_steps_keep_their_form(V):
    """Steps captured with the table and replayed among hot calls that would
    change the form: the table's chain."""
    import torch
    tab = I.eam_tables(I.multi_eam_params(2, dens_scale=(1.0, 1.25)))
    lat = I.bcc_lattice(48, 48, 48)
    R = 8
    types = np.stack([I.multi_random_types(lat.n, [lat.n // 3], seed=r) for r in range(R)])
    s = torch.cuda.Stream()
    args = (lat, types, tab, [-1.5], 0.0, 20000.0)
    g = V.Multi(*args, c0=0.3, seed_r=np.arange(R, dtype=np.uint64), stream=s)
    h = V.Multi(*args, c0=0.3, seed_r=np.arange(R, dtype=np.uint64))
    h.set_table(1)
    g.steps(2)
    graph = torch.cuda.CUDAGraph()
    s.synchronize()
    with torch.cuda.graph(graph, stream=s, capture_error_mode="thread_local"):
        g.steps(6)
    n = 2
    for _ in range(4):
        with torch.cuda.stream(s):
            graph.replay()
        g.observables(0)
        g.steps(256)
        g.observables(0)
        n += 6 + 256
    with torch.cuda.stream(s):
        graph.replay()
    h.steps(n + 6)
    for r in range(R):
        assert np.array_equal(g.types(r), h.types(r))
        assert g.observables(r)["flips"] == h.observables(r)["flips"] > n * 500
    del graph
    g.close()
    h.close()
