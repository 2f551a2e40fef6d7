"""The resident forms a context runs by default (csrc/kernels_cluster.cu),
against the oracle a stretch at a time: species bit for bit, counters exactly.
Sizes where they can go wrong: rows whose trials do not fill a word of four,
one word per row, tiles of two and three rows, several groups of trials per
thread, a single trial and more trials than threads per step, both
compile-time shell tables and the runtime one, both basis sites, stretches
below and above the shortest one that runs resident."""
import numpy as np
import pytest

import oracle as O
from paper_1012_5082_gb300 import inputs as I
from _pair import Lockstep

pytestmark = pytest.mark.gpu
KT = I.KB_EV


@pytest.fixture(scope="module")
def V():
    from paper_1012_5082_gb300 import vcsgc
    return vcsgc


def _tables(name):
    if name == "ising":
        return I.ising_tables()
    return I.eam_tables(I.EAMParams(rc=4.4, r_in=4.2)) if name == "three shells" else I.eam_tables()


@pytest.mark.parametrize("kind,cells,sched,alloy", [
    ("sublattice", (8, 8, 8), (4, 4, 4), "eam"),
    ("sublattice", (12, 8, 16), (4, 4, 4), "eam"),
    ("sublattice", (20, 12, 24), (4, 4, 4), "eam"),
    ("sublattice", (28, 36, 8), (4, 4, 4), "eam"),
    ("sublattice", (44, 48, 40), (4, 4, 4), "eam"),
    ("sublattice", (24, 20, 12), (4, 4, 4), "ising"),
    ("sublattice", (60, 64, 52), (4, 4, 4), "ising"),
    ("sublattice", (25, 10, 15), (5, 5, 5), "eam"),
    ("blocks", (10, 10, 10), (5, 5, 5, 2, 2, 2), "eam"),
    ("blocks", (16, 8, 24), (4, 4, 4, 2, 2, 2), "eam"),
    ("blocks", (40, 80, 80), (4, 4, 4, 2, 2, 2), "eam"),
    ("blocks", (20, 30, 40), (5, 5, 5, 2, 2, 2), "ising"),
    ("blocks", (16, 24, 8), (4, 4, 4, 2, 2, 2), "three shells"),
    ("overlap", (20, 30, 20), (10, 10, 10, 4, 4, 4), "eam"),
])
def test_resident_steps_match_the_oracle(V, kind, cells, sched, alloy):
    tab, lat = _tables(alloy), I.bcc_lattice(*cells)
    T, kappa = (1000.0, 10.0) if alloy == "ising" else (900.0, 1.0)
    c0, dmu0 = (0.5, 0.0) if alloy == "ising" else (0.1, -2.1)
    phi = dmu0 - 2.0 * kappa * KT * T * c0
    types = I.random_types(lat.n, int(c0 * lat.n), seed=lat.n)
    seeds = [lat.n + 1, lat.n + 2]
    skind = {"sublattice": V.SCHED_SUBLATTICE, "blocks": V.SCHED_BLOCKS, "overlap": V.SCHED_OVERLAP}[kind]
    g = V.Context(lat, np.tile(types, 2), tab, 0.0, kappa, T, schedule=skind, sched=sched, n_replicas=2,
                  phi_r=np.full(2, phi), c0_r=np.full(2, c0), seed_r=np.array(seeds, np.uint64))
    orcs = []
    for s in seeds:
        o = O.System(lat, types, tab)
        o.set_params(phi, kappa, T, c0=c0, seed=s)
        if kind == "sublattice":
            o.schedule_sublattice(cells, sched)
        elif kind == "blocks":
            o.schedule_blocks(cells, sched[:3], sched[3:])
        else:
            o.schedule_overlap(cells, sched[:3], sched[3:])
        orcs.append(o)
    ls = Lockstep(orcs, g)
    for n in (3, 64, 8, 7, 130):
        ls.advance(n)
    assert sum(g.observables(r)["flips"] for r in range(2)) > 0
    ls.close()
    g.close()
