"""Read-out into the caller's memory (csrc/readout.h): fresh, used, pinned and
unaligned buffers of a page and more hold the device's values, and nothing
around them changes."""
import ctypes as C

import numpy as np
import pytest

from paper_1012_5082_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cells", [(6, 6, 6), (16, 16, 9), (30, 31, 33)])
def test_read_out_into_any_buffer(cells):
    import torch

    from paper_1012_5082_gb300 import vcsgc as V
    lat = I.bcc_lattice(*cells)
    types = I.random_types(lat.n, lat.n // 3, seed=1)
    g = V.Context(lat, types, I.eam_tables(), -2.0, 10.0, 700.0, schedule=V.SCHED_SPATIAL, sched=(2, 2, 2, 2, 2, 2))
    g.set_velocities(I.maxwell_velocities(types, 600.0, seed=3))
    want = [np.array(a) for a in g.md_state()]
    for a, b in zip(want[:3], (lat.x, lat.y, lat.z)):
        assert np.array_equal(a, b)
    n8 = 8 * lat.n
    for lead in (0, 8, 4088, 65528):
        raw = [np.full(lead + n8 + 64, 0xA5, np.uint8) for _ in range(5)]
        pinned = torch.full((lead + n8 + 64,), 0xA5, dtype=torch.uint8, pin_memory=True).numpy()
        raw.append(pinned)
        ptr = [C.c_void_p(a.ctypes.data + lead) for a in raw]
        assert V.lib().vcsgc_get_md(g.h, *ptr) == 0
        for a, w in zip(raw, want):
            assert np.array_equal(a[lead:lead + n8].view(np.float64), w)
            assert (a[:lead] == 0xA5).all() and (a[lead + n8:] == 0xA5).all()
        t = np.full(lead + lat.n + 1, 0xA5, np.uint8)
        assert V.lib().vcsgc_get_types(g.h, 0, C.c_void_p(t.ctypes.data + lead)) == 0
        assert np.array_equal(t[lead:-1], types) and t[-1] == 0xA5 and (t[:lead] == 0xA5).all()
    g.close()
