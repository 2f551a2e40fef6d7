"""The neighbour list build (csrc/kernels_nbr.cu): rows and their order, against
a list made here pair by pair.  Sizes where the build can go wrong: three, four
and five cells per axis (faces on every side, no interior cell, one), empty
cells, cells of more atoms than a block takes at a time, neighbourhoods larger
than the staging buffer, rows cut at K; and the domain sort of the spatial
schedule below and above the bins it ranks in shared memory."""
import numpy as np
import pytest

from paper_1012_5082_gb300 import inputs as I

pytestmark = pytest.mark.gpu
RL = 5.6


def _rows(pos, box, rl):
    """Rows in the documented order: the 27 cells (x fastest), ascending index
    in each; FP32 distances as the list's criterion, with pairs so near its
    edge that rounding decides left out of `sure`."""
    n, nc = len(pos[0]), [int(b / rl) for b in box]
    c = [np.minimum((p / b * k).astype(int), k - 1) for p, b, k in zip(pos, box, nc)]
    bins = {}
    for i, q in enumerate(zip(*c)):
        bins.setdefault(q, []).append(i)
    margin = rl + 0.01 + 1e-6 * max(box)
    rows, edge = [], []
    P = np.stack(pos, 1)
    for i in range(n):
        cand = []
        for oz in (-1, 0, 1):
            for oy in (-1, 0, 1):
                for ox in (-1, 0, 1):
                    cand += bins.get(tuple((c[a][i] + o) % nc[a] for a, o in enumerate((ox, oy, oz))), [])
        cand = np.array([j for j in cand if j != i], int)
        d = P[cand] - P[i] if len(cand) else np.zeros((0, 3))
        d -= box * np.rint(d / box)
        r = np.sqrt((d * d).sum(1))
        rows.append(cand[r < margin - 1e-4])
        edge.append(set(cand[np.abs(r - margin) <= 1e-4].tolist()))
    return rows, edge


def _positions(name):
    rng = np.random.default_rng(len(name))
    if name == "clump":  # one dense cluster in a box of five cells: most cells empty
        box = np.array([28.5, 30.0, 33.0])
        return [14.0 + rng.uniform(-2.4, 2.4, 1300) for _ in range(3)], box
    if name == "corner clump":
        box = np.array([17.0, 23.0, 40.0])
        return [(rng.uniform(-2.0, 2.0, 1200)) % b for b in box], box
    box = {"3 x 3 x 3": [17.0, 18.0, 17.5], "4 x 3 x 5": [23.0, 17.0, 29.0], "6 x 5 x 7": [34.0, 29.0, 40.0]}[name]
    box = np.array(box)
    n = int(0.085 * box.prod())
    return [rng.uniform(0, b, n) for b in box], box


@pytest.mark.parametrize("name", ["3 x 3 x 3", "4 x 3 x 5", "6 x 5 x 7", "clump", "corner clump"])
def test_rows_and_their_order(name):
    import torch

    from paper_1012_5082_gb300 import vcsgc as V
    pos, box = _positions(name)
    n = len(pos[0])
    rows, edge = _rows(pos, box, RL)
    most = max(len(r) + len(e) for r, e in zip(rows, edge))
    d = [torch.tensor(p, dtype=torch.float64, device="cuda") for p in pos]
    for K in (most + 5, most // 2):
        nbr = torch.full((n, K), -7, dtype=torch.int32, device="cuda")
        cnt = torch.full((n,), -7, dtype=torch.int32, device="cuda")
        torch.cuda.synchronize()
        rc = V.vcsgc_neighbour_list_noalloc(n, *(p.data_ptr() for p in d), box, RL, K, nbr.data_ptr(), cnt.data_ptr(), None)
        assert (rc == 0) == (K > most)
        nb, ct = nbr.cpu().numpy(), cnt.cpu().numpy()
        for i in range(n):
            got = [j for j in nb[i, :ct[i]] if j not in edge[i]]
            assert (nb[i, ct[i]:] == -1).all()
            if ct[i] < K or K > most:
                assert got == rows[i].tolist()
            else:
                assert got == rows[i][:len(got)].tolist() and len(set(nb[i].tolist())) == K


@pytest.mark.parametrize("cells,nb", [((8, 8, 8), 2), ((26, 27, 26), 2), ((18, 18, 18), 4)])
def test_domain_tables_after_a_cycle(cells, nb):
    """A cycle without MD rebuilds the spatial schedule on the device: the same
    chain as without the rebuild (18252 atoms / 8 boxes are ranked, 36504 / 8
    exceed the ranked size)."""
    from paper_1012_5082_gb300 import vcsgc as V
    lat = I.bcc_lattice(*cells)
    rng = np.random.default_rng(3)
    lat = I.Lattice(x=(lat.x + rng.uniform(-0.05, 0.05, lat.n)) % lat.box[0],
                    y=(lat.y + rng.uniform(-0.05, 0.05, lat.n)) % lat.box[1],
                    z=(lat.z + rng.uniform(-0.05, 0.05, lat.n)) % lat.box[2], box=lat.box.copy())
    order = rng.permutation(lat.n)  # atoms in no spatial order
    lat = I.Lattice(x=lat.x[order], y=lat.y[order], z=lat.z[order], box=lat.box)
    t = I.random_types(lat.n, lat.n // 10, seed=4)
    v = I.maxwell_velocities(t, 300.0, seed=5)
    got = []
    for device in (False, True):
        g = V.Context(lat, t, I.eam_tables(), -2.0, 1.0, 900.0, c0=0.1, schedule=V.SCHED_SPATIAL,
                      sched=(nb, nb, nb, 2, 2, 2), seed=9)
        g.set_velocities(v)
        if device:
            g.hybrid(1, 0, 60)
        else:
            g.steps(60)
        got.append((g.types(), g.observables()["flips"]))
        g.close()
    assert got[0][1] == got[1][1] > 0 and np.array_equal(got[0][0], got[1][0])
