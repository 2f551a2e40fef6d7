"""Performance cases of the VC-SGC library: the work its users have it do.

Each case is one call sequence of a production run through the public Python
binding (``paper_1012_5082_gb300.vcsgc``): advance a chain, a trajectory or the
learned stage by a stretch, then read the state a run writes out.  A state
keeps what such a program keeps between stretches (the context, pinned host
buffers); every pass continues the chain where the last one stopped.

Kinds of case
  rigid      rigid BCC lattice, one density function: period-4 sublattice,
             octant blocks or overlapping domains; EAM or the Ising lattice gas
  batch      rigid lattices of uneven sizes at a grid of (phi, T) points, plain
             or with the learned first stage (delayed acceptance)
  reembed    rigid lattice with f_B = 1.25 f_A, plain or delayed acceptance
  multi      K species, with or without species-dependent densities
  md         molecular dynamics of explicit positions
  hybrid     one hybrid cycle: MD, then MC on the positions it reached
  surrogate  features of every site, the network's forward pass, one gradient
"""
import functools
import itertools
import math

import numpy as np
import torch

from paper_1012_5082_gb300 import inputs as I
from paper_1012_5082_gb300 import vcsgc as V

DMU0_600K = -2.0194  # eV: driving force balanced on the random 2 % start at 600 K
T_MD = 700.0


def listed():
    rigid = dict(kind="rigid", alloy="eam", sched="sublattice", mixed=False)
    eight = dict(nx=80, ny=80, nz=80, replicas=8)
    return [
        # the smallest run: 2000 sites, one trial per colour step, as in parity
        # checks, pre-scans and teaching runs; launch and step latency count
        dict(rigid, name="parity_10", nx=10, ny=10, nz=10, replicas=1, sched="blocks", block=5, sweeps=1),
        # the paper's Ising set-up: 40^3 cells, 64 domains in octants
        dict(rigid, name="ising_40", alloy="ising", nx=40, ny=40, nz=40, replicas=1, sched="blocks", block=5,
             sweeps=1),
        # production: 1,024,000 sites at 8 phi values across the miscibility gap
        dict(rigid, **eight, name="rigid_80x8", sweeps=5),
        # the largest lattice, in the mixed-precision form
        dict(rigid, name="rigid_128x8_mixed", nx=128, ny=128, nz=128, replicas=8, mixed=True, sweeps=2),
        # 64 uneven lattices (24^3 to 48^3) at 64 (phi, T) points
        dict(kind="batch", name="batch_64", replicas=64, smallest=24, sweeps=4, delayed=False),
        # species-dependent densities: every trial re-embeds its neighbours
        dict(eight, kind="reembed", name="reembed_80x8", sched="sublattice", delayed=False, sweeps=5),
        # the same chain with the learned first stage
        dict(eight, kind="reembed", name="delayed_80x8", sched="sublattice", delayed=True, sweeps=5),
        # ternary alloy, one density function
        dict(eight, kind="multi", name="ternary_80x8", species=3, sweeps=5),
        # quaternary alloy with species-dependent densities
        dict(eight, kind="multi", name="quaternary_80x8", species=4, sweeps=5),
        # MD of 1.36 M atoms, Langevin at 700 K, FP64: the largest case
        dict(kind="md", name="md_25nm", shape="crystal", size=88, ensemble="langevin", mixed=False, steps=20),
        # the paper's hybrid scheme on a 10 nm nanocrystal: 20 MD steps, 0.1 N trials
        dict(kind="hybrid", name="hybrid_10nm", size=100, grains=6, mixed=False, steps=20),
        # sample generation and one training gradient of the learned stage
        dict(kind="surrogate", name="surrogate_48", nx=48, ny=48, nz=48, batch=4096),
    ]


def _log_int(rng, lo, hi, step=1):
    """An integer multiple of step in [lo, hi], spread over its logarithm."""
    v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return max(lo, min(hi, int(round(v / step)) * step))


def draw(rng):
    kind = rng.choice(["rigid", "rigid", "blocks", "batch", "reembed", "multi", "md", "md", "hybrid", "surrogate"])
    if kind == "rigid":
        c = {k: _log_int(rng, 16, 128, 4) for k in ("nx", "ny", "nz")}
        return dict(c, kind="rigid", alloy=rng.choice(["eam", "eam", "ising"]), sched="sublattice",
                    mixed=rng.random() < 0.3, replicas=rng.randint(1, 8), sweeps=rng.randint(2, 5))
    if kind == "blocks":
        b = rng.choice([4, 5, 7])
        m = 80 // (2 * b)
        # blocks of b cells in octants, an even number of them per axis
        c = {k: 2 * b * rng.randint(1, m) for k in ("nx", "ny", "nz")}
        return dict(c, kind="rigid", alloy=rng.choice(["eam", "ising"]), sched=rng.choice(["blocks", "overlap"]),
                    block=b, mixed=False, replicas=rng.randint(1, 4), sweeps=1)
    if kind == "batch":
        return dict(kind="batch", replicas=_log_int(rng, 6, 64), smallest=4 * rng.randint(3, 6),
                    sweeps=rng.randint(2, 5), delayed=rng.random() < 0.3)
    if kind == "reembed":
        sched = rng.choice(["sublattice", "sublattice", "blocks"])
        step, top = (4, 80) if sched == "sublattice" else (8, 48)
        c = {k: _log_int(rng, 16, top, step) for k in ("nx", "ny", "nz")}
        return dict(c, kind="reembed", sched=sched, block=4, delayed=sched == "sublattice" and rng.random() < 0.4,
                    replicas=rng.randint(1, 8), sweeps=2 if sched == "sublattice" else 1)
    if kind == "multi":
        c = {k: _log_int(rng, 16, 80, 4) for k in ("nx", "ny", "nz")}
        return dict(c, kind="multi", species=rng.choice([2, 3, 4]), replicas=rng.randint(1, 8),
                    sweeps=rng.randint(1, 3))
    if kind == "md":
        ens = rng.choice(["langevin", "langevin", "langevin", "nvt", "npt"])
        return dict(kind="md", shape="crystal", size=_log_int(rng, 9, 80), ensemble=ens,
                    mixed=ens != "npt" and rng.random() < 0.4, steps=rng.randint(10, 20))
    if kind == "hybrid":
        return dict(kind="hybrid", size=_log_int(rng, 46, 110), grains=rng.randint(2, 8),
                    mixed=rng.random() < 0.3, steps=rng.randint(5, 20))
    c = {k: _log_int(rng, 12, 64, 4) for k in ("nx", "ny", "nz")}
    return dict(c, kind="surrogate", batch=_log_int(rng, 500, 16384))


# ------------------------------------------------------------------ inputs
@functools.lru_cache(maxsize=None)
def _tables(name):
    if name == "ising":
        return I.ising_tables()
    if name == "eam":
        return I.eam_tables()
    if name == "zero_pressure":
        return I.eam_tables(I.npt_eam_params())
    if name == "f_b_1.25":
        return I.eam_tables(I.multi_eam_params(2, dens_scale=(1.0, 1.25)))
    if name == "ternary":
        return I.eam_tables(I.multi_eam_params(3))
    return I.eam_tables(I.multi_eam_params(4, dens_scale=(1.0, 1.25, 0.85, 1.1)))


@functools.lru_cache(maxsize=4)
def _lattice(nx, ny, nz):
    return I.bcc_lattice(nx, ny, nz)


def _phi(dmu0, kappa, T, c0):
    """phi with phi + 2 kappa kB T c0 = dmu0."""
    return dmu0 - 2.0 * kappa * I.KB_EV * T * np.asarray(c0, dtype=np.float64)


def _seeds(seed, n):
    return np.arange(n, dtype=np.uint64) + np.uint64(1000 * (int(seed) % 1_000_003) + 1)


def _host(n):
    """A pinned host buffer for the species read after each stretch."""
    return torch.empty(n, dtype=torch.uint8, pin_memory=torch.cuda.is_available())


def _linear_network(coef, const, rng):
    """Packed parameters of a 10-64-64-1 SiLU network that evaluates a linear
    function of the ten counts (silu(x) - silu(-x) = x carries each input
    through both layers), its other units small and random as in training."""
    top = np.array([8, 6, 12, 24, 8, 56, 48, 96, 192, 64], dtype=np.float64)
    W1, W2, w3 = rng.normal(0, 0.05, (64, 10)), rng.normal(0, 0.05, (64, 64)), rng.normal(0, 1e-5, 64)
    W1[:20], W2[:20], W2[:, :20] = 0.0, 0.0, 0.0
    for q in range(10):
        W1[2 * q, q], W1[2 * q + 1, q] = 1.0, -1.0
        W2[2 * q, 2 * q], W2[2 * q, 2 * q + 1] = 1.0, -1.0
        W2[2 * q + 1, 2 * q], W2[2 * q + 1, 2 * q + 1] = -1.0, 1.0
        w3[2 * q], w3[2 * q + 1] = coef[q] * top[q], -coef[q] * top[q]
    z = np.zeros(64)
    return np.concatenate([W1.ravel(), z, W2.ravel(), z, w3, [const]]).astype(np.float32)


def _shells():
    """(half-lattice offset, shell) of the 58 BCC neighbours within 5.3 A and
    the shell radii, a = 2.855 A."""
    hs = [h for h in itertools.product(range(-3, 4), repeat=3) if len({q & 1 for q in h}) == 1 and any(h)]
    d2 = sorted({sum(q * q for q in h) for h in hs if sum(q * q for q in h) <= 12})
    return [(h, d2.index(sum(q * q for q in h))) for h in hs if sum(q * q for q in h) <= 12], \
        [0.5 * 2.855 * math.sqrt(v) for v in d2]


def _fixed_density_coefs():
    """E(B) - E(A) of a site as c + sum_s g_s (B neighbours in shell s), one
    density function, from the closed forms."""
    p = I.EAMParams()
    offs, radii = _shells()
    z = [sum(1 for _, s in offs if s == q) for q in range(5)]
    aa, ab, bb = ([float(p.pair(q, r)[0]) for r in radii] for q in range(3))
    rho = sum(n * float(p.dens(0, r)[0]) for n, r in zip(z, radii))
    const = sum(n * (y - x) for n, x, y in zip(z, aa, ab)) + float(p.embed(1, rho)[0]) - float(p.embed(0, rho)[0])
    return np.array([x - 2 * y + w for x, y, w in zip(aa, ab, bb)]), const


# a linear fit of E(B) - E(A) on random 5 % alloys with f_B = 1.25 f_A (rms 1.1e-4 eV)
FIT_1_25 = ((-0.00936064, -0.00911355, 0.00890181, 0.0115398, 0.00757281, -0.0110778, -0.0165421, 0.000252865,
             0.000141791, 9.18164e-05), 1.51338)


def _surrogate(delayed, coef, const, seed):
    return V.Surrogate(_linear_network(coef, const, np.random.default_rng(seed + 77))) if delayed else None


@functools.lru_cache(maxsize=4)
def _nanocrystal(size, grains):
    return I.nanocrystal(float(size), grains, seed=1002)


def _shaken(lat, seed):
    """The same atoms with thermal displacements."""
    rng = np.random.default_rng(seed)
    x, y, z = (np.mod(q + rng.normal(0.0, 0.05, lat.n), lat.box[0]) for q in (lat.x, lat.y, lat.z))
    return I.Lattice(x=x, y=y, z=z, box=lat.box)


def _crystal(case, seed):
    """A periodic crystal with thermal displacements, species and velocities."""
    n = case["size"]
    lat = _shaken(_lattice(n, n, n), seed)
    types = I.random_types(lat.n, max(1, lat.n // 100), seed + 1)
    return lat, types, I.maxwell_velocities(types, T_MD, seed + 2)


def prepare(case, seed):
    k, seed = case["kind"], int(seed)
    st = dict(kind=k, case=dict(case))
    R = case.get("replicas", 1)
    sub = dict(schedule=V.SCHED_SUBLATTICE, sched=(4, 4, 4, 0, 0, 0))
    if k in ("rigid", "reembed", "multi", "surrogate"):
        lat = _lattice(case["nx"], case["ny"], case["nz"])
    if k == "rigid" or k == "reembed":
        b = case.get("block", 4)
        sched = {"sublattice": sub, "blocks": dict(schedule=V.SCHED_BLOCKS, sched=(b, b, b, 2, 2, 2)),
                 "overlap": dict(schedule=V.SCHED_OVERLAP, sched=(2 * b,) * 3 + (4, 4, 4))}[case["sched"]]
    if k == "rigid":
        if case["alloy"] == "ising":
            T, kappa, c0, dmu0, frac = 1000.0, 100.0, np.full(R, 0.5), 0.0, 0.5
        elif R == 1:
            T, kappa, c0, dmu0, frac = 700.0, 1000.0, np.full(R, 0.05), -2.27, 0.05
        else:
            T, kappa, c0, dmu0, frac = 600.0, 1000.0, 0.02 + np.arange(R) * 0.48 / 7, DMU0_600K, 0.02
        types = np.concatenate([I.random_types(lat.n, int(round(frac * lat.n)), seed + r) for r in range(R)])
        st["ctx"] = V.Context(lat, types, _tables(case["alloy"]), 0.0, kappa, T, n_replicas=R,
                              phi_r=_phi(dmu0, kappa, T, c0), c0_r=c0, seed_r=_seeds(seed, R),
                              precision=V.PREC_MIXED if case["mixed"] else V.PREC_FP64, **sched)
        st["host"] = _host(R * lat.n)
    elif k == "batch":
        L = [case["smallest"] + 4 * (r % 7) for r in range(R)]
        T = np.array([500.0 + 400.0 * ((r // 8) % 8) / 7.0 for r in range(R)])
        c0 = np.array([0.02 + (r % 8) * 0.48 / 7 for r in range(R)])
        types = [I.random_types(2 * n ** 3, int(round(0.02 * 2 * n ** 3)), seed + r) for r, n in enumerate(L)]
        st["ctx"] = V.Batch([(n, n, n) for n in L], types, _tables("eam"), _phi(DMU0_600K, 1000.0, T, c0), 1000.0, T,
                            c0_r=c0, seed_r=_seeds(seed, R))
        g, const = _fixed_density_coefs()
        st["net"] = _surrogate(case["delayed"], np.concatenate([g, np.zeros(5)]), const, seed)
        st["host"] = _host(sum(2 * n ** 3 for n in L))
    elif k == "reembed":
        types = np.concatenate([I.random_types(lat.n, int(0.05 * lat.n), seed + r) for r in range(R)])
        st["ctx"] = V.Context(lat, types, _tables("f_b_1.25"), -2.2, 100.0, 1200.0, c0=0.05, n_replicas=R,
                              seed_r=_seeds(seed, R), **sched)
        st["net"] = _surrogate(case["delayed"], *FIT_1_25, seed)
        st["host"] = _host(R * lat.n)
    elif k == "multi":
        K = case["species"]
        name, phi, kappa = {2: ("f_b_1.25", [-2.2], 100.0), 3: ("ternary", [-1.928, -1.628], 10.0),
                            4: ("quaternary", [-1.173, -2.037, 0.567], 10.0)}[K]
        types = np.stack([I.multi_random_types(lat.n, [int(0.05 * lat.n)] * (K - 1), seed + r) for r in range(R)])
        st["ctx"] = V.Multi(lat, types, _tables(name), phi, kappa, 1200.0, c0=0.05, seed_r=_seeds(seed, R))
    elif k == "md" or k == "hybrid":
        prec = V.PREC_MIXED if case["mixed"] else V.PREC_FP64
        if k == "md":
            lat, types, v = _crystal(case, seed)
            name = "eam" if case["ensemble"] == "langevin" else "zero_pressure"
            phi = -1.0
        else:
            lat = _shaken(_nanocrystal(case["size"], case["grains"]), seed + 3)
            types = I.random_types(lat.n, max(1, lat.n // 100), seed + 1)
            v = I.maxwell_velocities(types, T_MD, seed + 2)
            name, phi = "eam", float(_phi(-2.0, 1000.0, T_MD, 0.01))
        nb = 2 * int(lat.box[0] // 22.0)  # boxes wider than two cutoffs, an even number per axis
        st["ctx"] = V.Context(lat, types, _tables(name), phi, 1000.0, T_MD, c0=0.01, schedule=V.SCHED_SPATIAL,
                              sched=(nb, nb, nb, 2, 2, 2), dt=2.0, gamma=0.01, T_md=T_MD, seed=seed, md_seed=seed,
                              precision=prec)
        st["ctx"].set_velocities(v)
        if k == "md" and case["ensemble"] != "langevin":
            st["ctx"].set_ensemble(case["ensemble"], t_damp=100.0, p_damp=1000.0, p_ext_bar=0.0)
        if k == "hybrid":
            st["mc_steps"] = max(1, int(round(0.1 * lat.n / (nb ** 3 // 8))))
    else:
        types = I.random_types(lat.n, int(0.1 * lat.n), seed)
        st["ctx"] = V.Context(lat, types, _tables("eam"), -2.0, 1000.0, 600.0, c0=0.1, seed=seed, **sub)
        st["net"] = V.Surrogate(I.mlp_init(seed, out_bias=2.0))
    if k in ("batch", "reembed") and st["net"] is not None:
        st["ctx"].set_surrogate(st["net"])
    return st


def _chain(ctx, host):
    """Species and running observables of every replica."""
    types = ctx.types_all(host.numpy())
    o = ctx.observables_all()
    return dict(types=types, n_b=[q["n_b"] for q in o], flips=[q["flips"] for q in o],
                local=[q["local_accepts"] for q in o], accepted=[q["global_accepts"] for q in o],
                energy=np.array([q["energy"] for q in o]), mean_c=np.array([q["mean_c"] for q in o]))


def _pack(d):
    return {k: np.array(v) if isinstance(v, list) else v for k, v in d.items()}


def run(state):
    ctx, case, k = state["ctx"], state["case"], state["kind"]
    if k in ("rigid", "batch", "reembed"):
        ctx.sweep(case["sweeps"])
        return _pack(_chain(ctx, state["host"]))
    if k == "multi":
        ctx.sweep(case["sweeps"])
        o = [ctx.observables(r) for r in range(ctx.R)]
        return dict(types=[ctx.types(r) for r in range(ctx.R)], n=np.array([q["n"] for q in o]),
                    flips=np.array([q["flips"] for q in o]), local=np.array([q["local_accepts"] for q in o]),
                    energy=np.array([q["energy"] for q in o]), mean_c=np.array([q["mean_c"] for q in o]))
    if k == "md":
        ctx.md_steps(case["steps"])
        return dict(state=ctx.md_state())
    if k == "hybrid":
        ctx.hybrid(1, case["steps"], state["mc_steps"])
        o = ctx.observables()
        return dict(state=ctx.md_state(), types=ctx.types(), n_b=o["n_b"], flips=o["flips"], energy=o["energy"])
    X, Y = ctx.features()
    g = state["net"].forward(X)
    grad, loss = state["net"].grad(X[:case["batch"]], Y[:case["batch"]])
    return dict(features=X, target=Y, predicted=g, grad=grad, loss=loss)


# -------------------------------------------------------------------- work
def _sites(case):
    if case["kind"] == "batch":
        return sum(2 * (case["smallest"] + 4 * (r % 7)) ** 3 for r in range(case["replicas"]))
    if case["kind"] == "md":
        return 2 * case["size"] ** 3
    if case["kind"] == "hybrid":
        return int(2 * (case["size"] / 2.855) ** 3)
    return 2 * case["nx"] * case["ny"] * case["nz"] * case.get("replicas", 1)


def work(case):
    """Bytes: the state read once and written once.  Flops: a rigid-lattice
    trial sums its 58 neighbours per shell and forms a five-term dE; a
    re-embedding trial adds two table cubics for each of 59 sites; an MD step
    takes about 90 per pair (29 pairs per atom) over both passes."""
    k, n = case["kind"], _sites(case)
    if k in ("rigid", "batch"):
        return dict(bytes=2.0 * n, flops=80.0 * n * case["sweeps"])
    if k == "reembed" or (k == "multi" and case["species"] != 3):
        return dict(bytes=2.0 * n, flops=(2 * 59 * 8 + 80.0) * n * case["sweeps"])
    if k == "multi":
        return dict(bytes=2.0 * n, flops=80.0 * n * case["sweeps"])
    if k == "md":
        return dict(bytes=97.0 * n, flops=29.0 * 90.0 * n * case["steps"])
    if k == "hybrid":
        return dict(bytes=98.0 * n, flops=29.0 * 90.0 * n * case["steps"] + 0.1 * n * 58 * 60.0)
    return dict(bytes=n * (1.0 + 44 + 4), flops=n * 10400.0 + min(n, case["batch"]) * 31000.0)


# ------------------------------------------------- 64-bit reference values
def exact(case, seed):
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    if case["kind"] == "md" and case["ensemble"] == "langevin":
        return dict(state=[q.cpu().numpy() for q in _langevin(case, int(seed), dev)])
    if case["kind"] == "surrogate":
        return _learned(case, int(seed), dev)
    return None  # the outcome of a Markov chain: whole numbers, and energies that follow from them


def _learned(case, seed, dev):
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    n = 2 * nx * ny * nz
    t = torch.from_numpy(I.random_types(n, int(0.1 * n), seed)).to(dev).reshape(nz, ny, nx, 2).double()
    offs, _ = _shells()

    def shifted(f, h):
        """f at the site h half-lattice units away, for both bases."""
        out = torch.empty_like(f)
        for b in (0, 1):
            q = [b + c for c in h]
            out[..., b] = torch.roll(f[..., q[0] & 1], (-(q[2] >> 1), -(q[1] >> 1), -(q[0] >> 1)), (0, 1, 2))
        return out

    own = [torch.zeros_like(t) for _ in range(5)]
    for h, s in offs:
        own[s] += shifted(t, h)
    near = [sum(shifted(own[s], h) for h, sh in offs if sh == 0) for s in range(5)]
    near[0] = near[0] - 8 * t
    X = torch.stack([q.reshape(-1) for q in own + near], 1)
    g, const = _fixed_density_coefs()
    Y = X[:, :5] @ torch.tensor(g, device=dev) + const
    p = torch.tensor(I.mlp_init(seed, out_bias=2.0), device=dev).double().requires_grad_(True)
    W1, b1, W2, b2, w3, b3 = torch.split(p, [640, 64, 4096, 64, 64, 1])
    top = torch.tensor([8, 6, 12, 24, 8, 56, 48, 96, 192, 64.0], device=dev).double()

    def net(x):
        h = torch.nn.functional.silu((x / top) @ W1.reshape(64, 10).T + b1)
        h = torch.nn.functional.silu(h @ W2.reshape(64, 64).T + b2)
        return h @ w3 + b3

    m = case["batch"]
    with torch.no_grad():
        out = net(X)
    loss = ((net(X[:m]) - Y[:m]) ** 2).mean()
    grad, = torch.autograd.grad(loss, p)
    return dict(features=X, target=Y, predicted=out, grad=grad, loss=float(loss.detach()))


def _philox(ctr, key):
    """Philox4x32-10 of counters (four int64 tensors of 32-bit words)."""
    M = 0xFFFFFFFF
    c0, c1, c2, c3 = ctr
    k0, k1 = key

    def mul(a, b):
        lo = (b & 0xFFFF) * a  # below 2^48
        hi = (b >> 16) * a
        full = hi + (lo >> 16)
        return full >> 16, ((full << 16) | (lo & 0xFFFF)) & M

    for _ in range(10):
        h0, l0 = mul(0xD2511F53, c0)
        h1, l1 = mul(0xCD9E8D57, c2)
        c0, c1, c2, c3 = h1 ^ c1 ^ k0, l1, h0 ^ c3 ^ k1, l0
        k0, k1 = (k0 + 0x9E3779B9) & M, (k1 + 0xBB67AE85) & M
    return c0, c1, c2, c3


def _normals(step, n, tag, key, dev):
    i = torch.arange(n, device=dev, dtype=torch.int64)
    z = torch.zeros_like(i)
    w = _philox((z + (step & 0xFFFFFFFF), z, i, z + tag), key)
    u1, u2 = ((((w[q + 1] << 21) | (w[q] >> 11)).double() * 2.0 ** -53) for q in (0, 2))
    r = torch.sqrt(-2.0 * torch.log1p(-u1))
    return r * torch.cos(2.0 * math.pi * u2), r * torch.sin(2.0 * math.pi * u2)


def _hermite(v, d, h, j, t):
    """Value and derivative of the cubic Hermite interpolant on interval j."""
    a, b, da, db = v[j], v[j + 1], d[j] * h, d[j + 1] * h
    c2, c3 = 3 * (b - a) - 2 * da - db, 2 * (a - b) + da + db
    return a + t * (da + t * (c2 + t * c3)), (da + t * (2 * c2 + 3 * t * c3)) / h


def _pairs(pos, L, rl, dev):
    """Indices (i, j), each unordered pair closer than rl once."""
    nc = int(L // rl)
    cell = torch.clamp((pos / L * nc).long(), max=nc - 1)
    cid = (cell[:, 2] * nc + cell[:, 1]) * nc + cell[:, 0]
    order = torch.argsort(cid)
    count = torch.bincount(cid, minlength=nc ** 3)
    start = torch.cumsum(count, 0) - count
    cap = int(count.max())
    slot = torch.arange(len(pos), device=dev) - start[cid[order]]
    table = torch.full((nc ** 3, cap), -1, device=dev, dtype=torch.int64)
    table[cid[order], slot] = order
    g = torch.arange(nc, device=dev)
    out = []
    for dz, dy, dx in itertools.product((-1, 0, 1), repeat=3):
        if (dz, dy, dx) < (0, 0, 0):
            continue
        other = ((((g + dz) % nc)[:, None, None] * nc + ((g + dy) % nc)[None, :, None]) * nc
                 + ((g + dx) % nc)[None, None, :]).reshape(-1)
        for part in torch.arange(nc ** 3, device=dev).split(16384):
            a = table[part][:, :, None].expand(-1, -1, cap)
            b = table[other[part]][:, None, :].expand(-1, cap, -1)
            ok = (a >= 0) & (b >= 0)
            if (dz, dy, dx) == (0, 0, 0):
                ok &= a < b
            a, b = a[ok], b[ok]
            d = pos[b] - pos[a]
            d = d - L * torch.round(d / L)
            near = (d * d).sum(1) < rl * rl
            out.append((a[near], b[near]))
    return torch.cat([q[0] for q in out]), torch.cat([q[1] for q in out])


def _langevin(case, seed, dev):
    """BAOAB Langevin MD of the same start, in 64 bits."""
    lat, types, v = _crystal(case, seed)
    tab, L = _tables("eam"), float(lat.box[0])
    D = functools.partial(torch.as_tensor, dtype=torch.float64, device=dev)
    pair, dpair = torch.stack([D(q) for q in tab.pair]), torch.stack([D(q) for q in tab.dpair])
    f, df = D(tab.dens[0]), D(tab.ddens[0])
    emb, demb = torch.stack([D(q) for q in tab.embed]), torch.stack([D(q) for q in tab.dembed])
    x = torch.stack([D(q) for q in (lat.x, lat.y, lat.z)], 1)
    vel = torch.stack([D(q) for q in v], 1)
    t = torch.as_tensor(types, device=dev).long()
    n, skin = len(x), 0.6
    built, (pi, pj) = x.clone(), _pairs(x, L, tab.rc + skin, dev)

    def locate(r, h, knots):
        j = torch.clamp((r / h).long(), max=knots - 2)
        return j, r / h - j

    def forces(x):
        rho = torch.zeros(n, dtype=torch.float64, device=dev)
        kept = []
        for a, b in zip(pi.split(1 << 24), pj.split(1 << 24)):
            d = x[b] - x[a]
            d = d - L * torch.round(d / L)
            r = torch.sqrt((d * d).sum(1))
            m = r < tab.rc
            a, b, d, r = a[m], b[m], d[m], r[m]
            j, s = locate(r, tab.dr, tab.nr)
            w, dw = _hermite(f, df, tab.dr, j, s)
            rho.index_add_(0, a, w).index_add_(0, b, w)
            q = (t[a] + t[b]) * tab.nr + j
            kept.append((a, b, d / r[:, None], dw, _hermite(pair.reshape(-1), dpair.reshape(-1), tab.dr, q, s)[1]))
        j, s = locate(rho, tab.drho, tab.nrho)
        dF = _hermite(emb.reshape(-1), demb.reshape(-1), tab.drho, t * tab.nrho + j, s)[1]
        F = torch.zeros_like(x)
        for a, b, e, dw, dp in kept:
            g = ((dF[a] + dF[b]) * dw + dp)[:, None] * e
            F.index_add_(0, a, g).index_add_(0, b, g, alpha=-1.0)
        return F

    im = (I.FTM / D([I.MASS_A, I.MASS_B]))[t][:, None]
    h, c1 = 1.0, math.exp(-0.01 * 2.0)
    sig = math.sqrt(1.0 - c1 * c1) * torch.sqrt(I.KB_EV * T_MD * im)
    key = (seed & 0xFFFFFFFF, (seed >> 32) & 0xFFFFFFFF)
    F = forces(x)
    for step in range(case["steps"]):
        vel = vel + h * F * im
        x = x + h * vel
        z0, z1 = _normals(step, n, 3, key, dev)
        z2, _ = _normals(step, n, 4, key, dev)
        vel = c1 * vel + sig * torch.stack([z0, z1, z2], 1)
        x = torch.remainder(x + h * vel, L)
        d = x - built
        d = d - L * torch.round(d / L)
        if float((d * d).sum(1).max()) > 0.25 * skin * skin:
            built, (pi, pj) = x.clone(), _pairs(x, L, tab.rc + skin, dev)
        F = forces(x)
        vel = vel + h * F * im
    return [x[:, 0], x[:, 1], x[:, 2], vel[:, 0], vel[:, 1], vel[:, 2]]
