"""Colour steps of three and four species (csrc/kernels_multi.cu), a stretch at a
time against the oracle, at sizes where the per-site entries, the split of a
trial over two lanes, the fold of a step by a block of its own and the wide
reads of a step's sums can go wrong: one period per axis, uneven axes, periods
other than four, blocks with one trial, half-filled warps, several replicas,
stretches of one step, and reads between them."""
import numpy as np
import pytest

import oracle as O
from paper_1012_5082_gb300 import inputs as I

pytestmark = pytest.mark.gpu

SPECIES = {
    3: [((1.0, 1.0, 1.0), [-1.928, -1.628]), ((1.0, 1.2, 0.9), [-2.1, -1.4])],
    4: [((1.0, 1.0, 1.0, 1.0), [-1.9, -1.7, -1.8]), ((1.0, 1.25, 0.85, 1.1), [-1.173, -2.037, 0.567])],
}


CASES = [(K, q, *c) for c in [((4, 4, 4), (4, 4, 4), 2), ((8, 4, 12), (4, 4, 4), 3), ((10, 5, 15), (5, 5, 5), 1),
                              ((12, 8, 10), (6, 4, 5), 1)] for K in (3, 4) for q in (0, 1)]


@pytest.mark.parametrize("K,reembed,cells,period,R", CASES + [(4, 1, (16, 16, 20), (4, 4, 4), 1)])
def test_steps_match_the_oracle(K, reembed, cells, period, R):
    from paper_1012_5082_gb300 import vcsgc as V
    ds, phi = SPECIES[K][reembed]
    tab = I.eam_tables(I.multi_eam_params(K, dens_scale=ds))
    lat = I.bcc_lattice(*cells)
    kappa, T, c0 = 0.05, 1200.0, 0.05
    types = np.stack([I.multi_random_types(lat.n, [max(1, int(c0 * lat.n))] * (K - 1), seed=r + 7) for r in range(R)])
    seeds = np.arange(R, dtype=np.uint64) + np.uint64(lat.n)
    g = V.Multi(lat, types, tab, phi, kappa, T, c0=c0, seed_r=seeds, period=period)
    orcs = []
    for r in range(R):
        o = O.MultiSystem(lat, types[r], tab)
        o.set_params(phi, [kappa] * (K - 1), T, c0=[c0] * (K - 1), seed=int(seeds[r]))
        o.schedule_sublattice(cells, period)
        orcs.append(o)
    flips = 0
    for n in (1, 1, 6, 64, 70):
        g.steps(n)
        for r, o in enumerate(orcs):
            o.parallel_steps(n)
            og, oo = g.observables(r), o.obs()
            assert oo["near_ties"] == og["near_ties"] == 0
            assert np.array_equal(g.types(r), o.types), (n, r)
            for k in ("trials", "local_accepts", "global_trials", "global_accepts", "flips", "steps"):
                assert og[k] == oo[k], (n, r, k, og[k], oo[k])
            assert og["n"] == oo["n"]
            for a in range(K):
                assert abs(og["mean_c"][a] * og["steps"] - oo["sum_c"][a]) < 1e-12 * oo["steps"]
            # a step's dE in FP64 and fixed point: 1e-9 of the total
            assert abs(og["energy"] - oo["energy"]) <= 1e-9 * abs(oo["energy"])
    for r, o in enumerate(orcs):
        e = o.energy_full()
        assert abs(g.energy(r) - e) <= 1e-12 * abs(e)
        flips += g.observables(r)["flips"]
    assert flips > 0
    g.close()
