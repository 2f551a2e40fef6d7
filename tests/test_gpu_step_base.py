"""The chain's position (step base, colour table, pending commit) across the
forms of the colour step: after a resident call the per-step launch goes on
from the device's own base, so a caller may capture steps into a graph of its
own and replay it, and the base is 64 bits everywhere."""
import struct

import numpy as np
import pytest

import oracle as O
from paper_1012_5082_gb300 import inputs as I

pytestmark = pytest.mark.gpu
T, KAPPA, C0, PHI = 900.0, 1.0, 0.1, -2.2
SCHED = {"sublattice": ((12, 8, 16), (4, 4, 4)), "blocks": ((16, 8, 24), (4, 4, 4, 2, 2, 2))}


@pytest.fixture(scope="module")
def V():
    from paper_1012_5082_gb300 import vcsgc
    return vcsgc


def _context(V, kind, **kw):
    cells, sched = SCHED[kind]
    lat, tab = I.bcc_lattice(*cells), I.eam_tables()
    types = I.random_types(lat.n, int(C0 * lat.n), seed=3)
    g = V.Context(lat, np.tile(types, 2), tab, PHI, KAPPA, T, c0=C0, n_replicas=2, seed_r=np.array([5, 6], np.uint64),
                  schedule=V.SCHED_SUBLATTICE if kind == "sublattice" else V.SCHED_BLOCKS, sched=sched, **kw)
    return lat, tab, types, g


def _oracles(kind, lat, tab, types):
    cells, sched = SCHED[kind]
    out = []
    for seed in (5, 6):
        o = O.System(lat, types, tab)
        o.set_params(PHI, KAPPA, T, c0=C0, seed=seed)
        if kind == "sublattice":
            o.schedule_sublattice(cells, sched)
        else:
            o.schedule_blocks(cells, sched[:3], sched[3:])
        out.append(o)
    return out


def _agree(g, orcs):
    for r, o in enumerate(orcs):
        oo, og = o.obs(), g.observables(r)
        assert oo["near_ties"] == 0
        assert np.array_equal(g.types(r), o.types)
        for k in ("n_b", "steps", "trials", "local_accepts", "global_accepts", "flips"):
            assert oo[k] == og[k], (r, k, oo[k], og[k])


@pytest.mark.parametrize("kind,shape", [("sublattice", None), ("blocks", None), ("sublattice", (1, 256, 2))])
def test_captured_steps_replay_after_resident_ones(V, kind, shape):
    """In the default form, and in form 1 asked for: a capture takes the
    per-step launch."""
    import torch
    s = torch.cuda.Stream()
    lat, tab, types, g = _context(V, kind, stream=s)
    if shape:
        g.set_launch(*shape)
    orcs = _oracles(kind, lat, tab, types)
    g.steps(23)  # resident
    graph = torch.cuda.CUDAGraph()
    s.synchronize()
    with torch.cuda.graph(graph, stream=s, capture_error_mode="thread_local"):
        g.steps(4)
    for _ in range(3):
        with torch.cuda.stream(s):
            graph.replay()
    s.synchronize()
    for o in orcs:
        o.parallel_steps(23 + 3 * 4)
    _agree(g, orcs)
    for n in (5, 40, 3):  # and on, in both forms
        g.steps(n)
        for o in orcs:
            o.parallel_steps(n)
        _agree(g, orcs)
    del graph
    g.close()


@pytest.mark.parametrize("kind", SCHED)
def test_resident_steps_follow_a_replay(V, kind):
    """A replay leaves a commit pending that the host has not seen: the next
    call, resident or a read, applies it."""
    import torch
    s = torch.cuda.Stream()
    lat, tab, types, g = _context(V, kind, stream=s)
    orcs = _oracles(kind, lat, tab, types)
    graph = torch.cuda.CUDAGraph()
    s.synchronize()
    with torch.cuda.graph(graph, stream=s, capture_error_mode="thread_local"):
        g.steps(5)
    g.types(0)  # nothing has run: no pending commit for the host
    with torch.cuda.stream(s):
        graph.replay()
        graph.replay()
    g.steps(30)  # resident
    for o in orcs:
        o.parallel_steps(2 * 5 + 30)
    _agree(g, orcs)
    with torch.cuda.stream(s):
        graph.replay()
    for o in orcs:
        o.parallel_steps(5)
    _agree(g, orcs)
    del graph
    g.close()


# ------------------------------------------------------------ 64-bit steps
def _move_base(path, base, n_replicas):
    """The checkpoint's chain moved to step `base`: the running states' next
    and last finalised steps and the step base."""
    b = bytearray(open(path, "rb").read())
    n, _, _, _, _, rs_bytes, _, _ = struct.unpack_from("<8q", b, 8)
    rs0 = 8 + 64 + 8 * n_replicas + n * n_replicas
    for r in range(n_replicas):
        struct.pack_into("<2q", b, rs0 + r * rs_bytes + 8, base, base - 1)
    struct.pack_into("<q", b, rs0 + n_replicas * rs_bytes, base)
    open(path, "wb").write(b)


@pytest.mark.parametrize("base", [2 ** 31 - 30, 2 ** 32 - 30, 3 * 2 ** 32 + 2 ** 31 + 7])
@pytest.mark.parametrize("kind", SCHED)
def test_bases_beyond_32_bits(V, tmp_path, kind, base):
    """Resident and per-step calls in turn across a 2^31 or 2^32 boundary give
    the chain that the per-step launch alone gives."""
    path = str(tmp_path / "chain")
    _, _, _, g = _context(V, kind)
    g.steps(2)
    g.save(path)
    g.close()
    _move_base(path, base, 2)
    out = []
    for mixed in (True, False):
        _, _, _, g = _context(V, kind)
        g.load(path)
        if not mixed:
            g.set_launch(0, 128, 1)
        for n in (16, 3, 9, 1, 70, 5):
            g.steps(n)
        out.append([(g.types(r), g.observables(r)) for r in range(2)])
        g.close()
    for (ta, oa), (tb, ob) in zip(*out):
        assert np.array_equal(ta, tb)
        for k in ("n_b", "steps", "trials", "local_accepts", "global_accepts", "flips", "near_ties"):
            assert oa[k] == ob[k], k
        assert oa["flips"] > 0


@pytest.mark.parametrize("ran", [1, 2, 4])
def test_load_into_a_context_that_has_run(V, tmp_path, ran):
    """A checkpoint continues the same chain whether the context it is loaded
    into is fresh or has run per-step calls of its own."""
    path = str(tmp_path / "chain")
    lat, tab, types, g = _context(V, "sublattice")
    g.steps(20)
    g.save(path)
    g.close()
    orcs = _oracles("sublattice", lat, tab, types)
    for o in orcs:
        o.parallel_steps(20 + 5)
    _, _, _, g = _context(V, "sublattice")
    g.steps(ran)
    g.load(path)
    g.steps(5)
    _agree(g, orcs)
    g.close()
