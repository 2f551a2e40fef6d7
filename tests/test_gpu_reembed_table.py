"""Species-dependent densities on the period-q sublattice: the re-embedding
table the colour steps read and the commit keeps up to date (kernels_multi.cu,
dtab), and the count-based densities and energies of the five-shell lattice
(kernels_nbr.cu, k_shell_state), against the oracle at sizes where the wraps
and remainders can go wrong: one period per axis, one place per class, uneven
axes, periods other than four, several replicas."""
import numpy as np
import pytest

import oracle as O
from paper_1012_5082_gb300 import inputs as I
from _pair import Lockstep

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def V():
    from paper_1012_5082_gb300 import vcsgc
    return vcsgc


@pytest.mark.parametrize("cells,period,R", [
    ((4, 4, 4), (4, 4, 4), 2), ((8, 4, 12), (4, 4, 4), 3), ((8, 12, 16), (4, 4, 4), 2), ((20, 8, 12), (4, 4, 4), 1),
    ((28, 16, 8), (4, 4, 4), 2), ((10, 5, 15), (5, 5, 5), 2), ((12, 8, 10), (6, 4, 5), 1), ((40, 44, 36), (4, 4, 4), 1),
])
def test_table_steps_match_the_oracle(V, cells, period, R):
    lat = I.bcc_lattice(*cells)
    tab = I.eam_tables(I.multi_eam_params(2, dens_scale=(1.0, 1.25)))
    types = I.random_types(lat.n, max(1, lat.n // 10), seed=lat.n)
    seeds = np.arange(R, dtype=np.uint64) + np.uint64(lat.n)
    T, kappa, c0, phi = 1200.0, 0.02, 0.1, -2.2
    g = V.Context(lat, np.tile(types, R), tab, phi, kappa, T, c0=c0, schedule=V.SCHED_SUBLATTICE, sched=period,
                  n_replicas=R, seed_r=seeds)
    orcs = []
    for s in seeds:
        o = O.System(lat, types, tab)
        o.set_params(phi, kappa, T, c0=c0, seed=int(s))
        o.schedule_sublattice(cells, period)
        orcs.append(o)
    ls = Lockstep(orcs, g)
    for n in (1, 5, 64, 130):
        ls.advance(n)
    for r in range(R):
        o = orcs[r]
        # densities: sums of 58 values of order 1 (15 in all), rounded once each
        assert np.max(np.abs(g.rho(r) - o.rho)) <= 58 * 15.5 * 2.0 ** -52 * 4
        assert abs(g.energy(r) - o.energy_full()) <= 1e-12 * abs(o.energy_full())
    assert sum(g.observables(r)["flips"] for r in range(R)) > 0
    ls.close()
    g.close()
