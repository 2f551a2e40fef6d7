"""The cluster sizes a context offers follow the shared memory the kernel uses:
where the default form runs a size on the five-shell table, that size can be
asked for."""
import numpy as np
import pytest

from paper_1012_5082_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def test_sizes_of_128_cubed():
    """128^3: 8 CTAs hold 68 x 36 rows of 9 words with their halos, 96 KB with
    their trials, and 4096 trials each; 4 CTAs would hold 8192 trials, more than a
    CTA's sums take."""
    from paper_1012_5082_gb300 import vcsgc as V
    lat = I.bcc_lattice(128, 128, 128)
    types = I.random_types(lat.n, lat.n // 20, seed=1)
    a, b = (V.Context(lat, types, I.eam_tables(), -2.0, 1.0, 900.0, c0=0.05, seed=4) for _ in range(2))
    assert a.cluster_sizes() == [8, 16]
    for block in (256, 512):
        a.set_launch(1, block, 8)
        a.steps(24)
    b.set_launch(0, 128, 1)
    b.steps(48)
    oa, ob = a.observables(), b.observables()
    assert np.array_equal(a.types(), b.types())
    for k in ("local_accepts", "global_accepts", "flips", "n_b"):
        assert oa[k] == ob[k]
    a.close()
    b.close()
