"""The half-list passes of the MD forces (csrc/kernels_md.cu) at the sizes where
their split can go wrong: atom counts that fill no warp, both sides of the
atom count at which an atom gets 4 lanes instead of 16, rows cut by the box
faces on every side, one density function for both species and two, the
virial in the same pass, and mixed precision."""
import numpy as np
import pytest

import oracle as O
from paper_1012_5082_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def V():
    from paper_1012_5082_gb300 import vcsgc
    return vcsgc


def _pair(V, cells, dens_b, prec):
    tab = I.eam_tables(I.EAMParams(dens_scale=(1.0, dens_b)))
    lat = I.bcc_lattice(*cells)
    rng = np.random.default_rng(lat.n)
    # a shift of a third of a cell puts layers on both sides of every face
    q = [(a + 0.95 + rng.uniform(-0.12, 0.12, lat.n)) % L for a, L in zip((lat.x, lat.y, lat.z), lat.box)]
    lat = I.Lattice(x=q[0], y=q[1], z=q[2], box=lat.box.copy())
    t = I.random_types(lat.n, lat.n // 3, seed=5)
    g = V.Context(lat, t, tab, -2.0, 10.0, 700.0, schedule=V.SCHED_SPATIAL, sched=(2, 2, 2, 2, 2, 2), precision=prec)
    return O.System(lat, t, tab), g, lat


SIZES = [(6, 6, 6), (7, 6, 9), (11, 13, 7), (21, 22, 21), (23, 21, 22)]


@pytest.mark.parametrize("dens_b", [1.0, 1.25])
@pytest.mark.parametrize("cells", SIZES)
def test_forces_energy_and_pressure(V, cells, dens_b):
    """About 60 terms of a few eV/A per atom, each good to some 2^-50: forces
    within 1e-10 eV/A; pressure and energy are sums over all pairs, within
    1e-10 relative."""
    orc, g, lat = _pair(V, cells, dens_b, V.PREC_FP64)
    so, sg = orc.ensemble_state(), g.ensemble_state()
    for k in ("potential", "pressure_bar"):
        assert abs(sg[k] - so[k]) <= 1e-10 * abs(so[k]) + 1e-9, (k, sg[k], so[k])
    Fg, Fo = g.forces(), orc.forces()
    for a in range(3):
        assert np.max(np.abs(Fg[a] - Fo[a])) < 1e-10
    # no net force: the two ends of every pair got the same term
    assert max(abs(F.sum()) for F in Fg) < 1e-9 * np.sqrt(lat.n)
    g.close()


@pytest.mark.parametrize("dens_b", [1.0, 1.25])
@pytest.mark.parametrize("cells", [SIZES[1], SIZES[3], SIZES[4]])
def test_forces_mixed(V, cells, dens_b):
    """FP32 pair terms (a few eV/A times 2^-24, about 60 of them)."""
    orc, g, lat = _pair(V, cells, dens_b, V.PREC_MIXED)
    Fg, Fo = g.forces(), orc.forces()
    for a in range(3):
        assert np.max(np.abs(Fg[a] - Fo[a])) < 2e-5
    g.close()


@pytest.mark.parametrize("dens_b", [1.0, 1.25])
@pytest.mark.parametrize("cells", [(6, 6, 6), (7, 6, 9), (36, 37, 38), (63, 64, 63)])
def test_pair_blocks_match_the_direct_passes(V, cells, dens_b):
    """MD passes leave each pair's distance for the force pass, in blocks of 2,
    4 or 16 atoms by size; the passes of a context that has not run MD do not.
    Same bounds as against the oracle."""
    orc, g, lat = _pair(V, cells, dens_b, V.PREC_FP64)
    want = [np.array(F) for F in g.forces()]
    p0 = g.ensemble_state()["pressure_bar"]
    g.minimize(ftol=1e-3, max_iter=0)
    got = g.forces()
    for a in range(3):
        assert np.max(np.abs(got[a] - want[a])) < 1e-10
    sg = g.ensemble_state()
    assert abs(sg["pressure_bar"] - p0) <= 1e-10 * abs(p0)
    got = g.forces()
    for a in range(3):
        assert np.max(np.abs(got[a] - want[a])) < 1e-10
    g.close()


def test_long_rows_take_several_lists(V):
    """A cutoff of 9 A: 132 pairs per half row, four atoms of a block overflow
    its list."""
    tab = I.eam_tables(I.EAMParams(rc=9.0, r_in=8.5))
    rng = np.random.default_rng(2)
    lat = I.bcc_lattice(37, 37, 38)
    q = [(x + rng.uniform(-0.05, 0.05, lat.n)) % b for x, b in zip((lat.x, lat.y, lat.z), lat.box)]
    lat = I.Lattice(x=q[0], y=q[1], z=q[2], box=lat.box.copy())
    t = I.random_types(lat.n, lat.n // 4, seed=1)
    orc = O.System(lat, t, tab)
    g = V.Context(lat, t, tab, -2.0, 10.0, 700.0, schedule=V.SCHED_SPATIAL, sched=(2, 2, 2, 2, 2, 2))
    g.minimize(ftol=1e-3, max_iter=0)
    Fg, Fo = g.forces(), orc.forces()
    for a in range(3):
        assert np.max(np.abs(Fg[a] - Fo[a])) < 1e-10
    g.close()


def test_coincident_atoms_are_an_error(V):
    """Two atoms at one place have no force direction: refused, not finite."""
    lat = I.bcc_lattice(6, 6, 6)
    x, y, z = (np.array(a) for a in (lat.x, lat.y, lat.z))
    x[101], y[101], z[101] = x[40], y[40], z[40]
    bad = I.Lattice(x=x, y=y, z=z, box=lat.box.copy())
    with pytest.raises(Exception):
        V.Context(bad, np.zeros(lat.n, np.uint8), I.eam_tables(), -2.0, 10.0, 700.0, schedule=V.SCHED_SPATIAL,
                  sched=(2, 2, 2, 2, 2, 2)).forces()
