"""Pair tables on either side of 2^19 intervals, where the MD passes change the
way they find a pair's interval: the same forces as with a smaller table to the
tables' accuracy, and an atom at no finite place is an error."""
import numpy as np
import pytest

from paper_1012_5082_gb300 import inputs as I

pytestmark = pytest.mark.gpu
TABLE_RANGE, NONFINITE = -3, -4


def _context(V, intervals):
    lat = I.bcc_lattice(7, 6, 9)
    rng = np.random.default_rng(1)
    q = [(a + rng.uniform(-0.1, 0.1, lat.n)) % L for a, L in zip((lat.x, lat.y, lat.z), lat.box)]
    lat = I.Lattice(x=q[0], y=q[1], z=q[2], box=lat.box.copy())
    t = I.random_types(lat.n, lat.n // 3, seed=5)
    g = V.Context(lat, t, I.eam_tables(I.EAMParams(nr=intervals + 1)), -2.0, 10.0, 700.0, schedule=V.SCHED_SPATIAL,
                  sched=(2, 2, 2, 2, 2, 2), dt=1.0)
    return lat, t, g


@pytest.mark.parametrize("intervals", [(1 << 19) - 1, 1 << 19])
def test_large_tables(intervals):
    """The half-list passes of a fresh context, and the pair blocks of one that
    runs MD.  Interpolation errors fall with h^3 in the derivative: below 1e-9
    eV/A with 20,000 intervals."""
    from paper_1012_5082_gb300 import vcsgc as V
    lat, t, g = _context(V, intervals)
    _, _, ref = _context(V, 20000)
    for run in (False, True):
        if run:
            for c in (g, ref):
                c.minimize(ftol=1e-3, max_iter=0)
        for a, b in zip(g.forces(), ref.forces()):
            assert np.max(np.abs(a - b)) < 1e-8
    ref.close()
    v = I.maxwell_velocities(t, 300.0, seed=2)
    v[1][17] = np.nan
    g.set_velocities(v)
    with pytest.raises(V.VcsgcError) as e:
        g.md_steps(1)
    assert e.value.code in (TABLE_RANGE, NONFINITE)
    g.close()
