"""Workloads of the Chebyshev random-probe tight-binding path, each one call (or one short sequence
of calls) of the public Python API as a user's program makes it.

The systems are those of the repository's own configurations: jittered copper-like fcc spheres with
the seed-5264 s/p/d Slater-Koster model (a = 3.61 A, 4 A cutoff, 11 electrons per atom), the
1-orbital simple-cubic open cluster with on-site disorder, and the periodic 9-orbital simple-cubic
lattice.  ``exact`` evaluates the same estimators with plain torch in 64 bits.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1812_05264_gb300 import _lib as L
from paper_1812_05264_gb300 import api

DEV = "cuda"
FCC_A, R0, DECAY, CUTOFF, ONSITE = 3.61, 2.55, 2.0, 4.0, (5.0, 10.0, 0.0)
SK_V = np.random.default_rng(5264).standard_normal(10)   # sss sps sds pps ppp pds pdp dds ddp ddd
BOUNDS_SEED = 0x5EED
M64 = (1 << 64) - 1


# ---- the cases ---------------------------------------------------------------------------------

def listed():
    return [
        # the plain-method test model: FP64 moments and mu of a 10^3 one-orbital cluster (smallest)
        {"name": "sc-energy-1000-fp64", "kind": "sc", "L": 10, "probes": 32, "order": 200},
        # one geometry step of a small cluster, positions in, energies and forces out
        {"name": "solver-147", "kind": "solver", "atoms": 147, "probes": 128, "order": 126, "kT": 0.5},
        # the 1,000-atom warm-dense workload, positions in, energies and forces out
        {"name": "solver-1000", "kind": "solver", "atoms": 1000, "probes": 256, "order": 126, "kT": 0.5},
        # what every new geometry of a large cluster needs first: neighbours, H, spectral bounds
        {"name": "setup-10000", "kind": "setup", "atoms": 10000},
        # chemical potential and observables from the moments of a near-ambient expansion
        {"name": "fermi-2476", "kind": "fermi", "states": 90000, "order": 2476, "kT": 0.025},
        # moments of the periodic 9-orbital lattice (every row full, panels beyond L2)
        {"name": "lattice-24-moments", "kind": "lattice", "L": 24, "probes": 512, "order": 128},
        # energies, sampled density matrix and forces of the 10,000-atom cluster (largest)
        {"name": "forces-10000", "kind": "forces", "atoms": 10000, "probes": 512, "order": 126, "kT": 0.5,
         "fp64": False},
        # many clusters of uneven size and temperature in one call
        {"name": "batch-16", "kind": "batch", "clusters": 16, "lo": 100, "hi": 1500, "probes": 128,
         "windowed": True},
        # probe counts that are no multiple of 128: quick, noisy estimates
        {"name": "forces-333-ragged", "kind": "forces", "atoms": 333, "probes": 100, "order": 250, "kT": 0.25,
         "fp64": False},
        # FP64 energies and forces, the reference precision, on a cluster one would check against
        {"name": "forces-200-fp64", "kind": "forces", "atoms": 200, "probes": 64, "order": 126, "kT": 0.5,
         "fp64": True},
        # direct random estimate of the density and energy-density matrices
        {"name": "direct-1000", "kind": "direct", "atoms": 1000, "probes": 256, "order": 126, "kT": 0.5},
        # local approximation with regions of 6 A
        {"name": "local-500", "kind": "local", "atoms": 500, "r_max": 6.0, "order": 126, "kT": 0.5},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the listed kinds, sizes spread over the ranges that they stand for."""
    kind = rng.choice(["sc", "solver", "solver", "setup", "fermi", "lattice", "forces", "forces", "batch",
                       "ragged", "fp64", "direct", "local"])
    kT = rng.choice([0.1, 0.25, 0.5])
    order = {0.1: 630, 0.25: 252, 0.5: 126}[kT] + rng.randint(-5, 5)
    wide = rng.choice([128, 256, 512])
    if kind == "sc":
        return {"kind": "sc", "L": rng.randint(6, 14), "probes": 4 * rng.randint(2, 16), "order": rng.randint(60, 400)}
    if kind == "solver":
        return {"kind": "solver", "atoms": _log_int(rng, 55, 2000), "probes": rng.choice([128, 256]),
                "order": rng.randint(100, 150), "kT": 0.5}
    if kind == "setup":
        return {"kind": "setup", "atoms": _log_int(rng, 100, 10000)}
    if kind == "fermi":
        return {"kind": "fermi", "states": _log_int(rng, 900, 90000), "order": _log_int(rng, 64, 2500),
                "kT": rng.choice([0.025, 0.1, 0.5])}
    if kind == "lattice":
        return {"kind": "lattice", "L": rng.randint(6, 22), "probes": wide, "order": rng.randint(60, 130)}
    if kind == "forces":
        return {"kind": "forces", "atoms": _log_int(rng, 100, 2000), "probes": wide, "order": order, "kT": kT,
                "fp64": False}
    if kind == "batch":
        return {"kind": "batch", "clusters": rng.randint(2, 16), "lo": 100, "hi": _log_int(rng, 200, 1500),
                "probes": rng.choice([128, 128, 256]), "windowed": rng.random() < 0.5}
    if kind == "ragged":
        return {"kind": "forces", "atoms": _log_int(rng, 30, 330), "probes": 4 * rng.randint(2, 31),
                "order": rng.randint(100, 220), "kT": 0.25, "fp64": False}
    if kind == "fp64":
        return {"kind": "forces", "atoms": _log_int(rng, 30, 400), "probes": 4 * rng.randint(2, 32),
                "order": rng.randint(64, 160), "kT": 0.5, "fp64": True}
    if kind == "direct":
        return {"kind": "direct", "atoms": _log_int(rng, 60, 2000), "probes": rng.choice([128, 256]),
                "order": rng.randint(100, 150), "kT": 0.5}
    return {"kind": "local", "atoms": _log_int(rng, 60, 600), "r_max": rng.uniform(4.0, 6.5),
            "order": rng.randint(64, 150), "kT": 0.5}


# ---- inputs --------------------------------------------------------------------------------------

def _fcc_sites(n):
    """The n fcc sites closest to the origin, in units of a/2, by (r^2, x, y, z)."""
    r = int(np.ceil((6.0 * n / np.pi) ** (1.0 / 3.0))) + 3
    g = np.arange(-r, r + 1)
    x, y, z = (v.ravel() for v in np.meshgrid(g, g, g, indexing="ij"))
    keep = (x + y + z) % 2 == 0
    x, y, z = x[keep], y[keep], z[keep]
    order = np.lexsort((z, y, x, x * x + y * y + z * z))[:n]
    return np.stack([x[order], y[order], z[order]], axis=1)


def _fcc(n, seed):
    pos = _fcc_sites(n) * (FCC_A / 2.0) + np.random.default_rng(seed).normal(0.0, 0.05, size=(n, 3))
    return torch.as_tensor(pos, device=DEV)


def _cubic(size):
    g = np.arange(size, dtype=np.float64)
    return np.stack([v.ravel() for v in np.meshgrid(g, g, g, indexing="ij")], axis=1)


def _lattice_model(seed):
    """Hopping blocks of the nine half directions of the periodic lattice, a band about 10 eV wide."""
    dirs = np.array([[1, 0, 0], [0, 1, 0], [0, 0, 1], [1, 1, 0], [1, -1, 0], [1, 0, 1], [1, 0, -1], [0, 1, 1],
                     [0, 1, -1]], dtype=np.float64)
    h = np.random.default_rng(seed).standard_normal((9, 9, 9)) * (10.0 / 52.6)
    return np.concatenate([dirs, -dirs]), np.concatenate([h, np.transpose(h, (0, 2, 1))])


def _sk_model():
    return api.Model(L.TBK_MODEL_SK, 9, sk_V=SK_V, r0=R0, decay=DECAY, onsite_spd=ONSITE)


def _batch(case, seed):
    """(atoms, order, kT, seed) of every cluster: sizes log-uniform and fixed by the case, temperatures
    in turn, orders as the error model gives them for this model's width."""
    n, lo, hi = case["clusters"], math.log(case["lo"]), math.log(case["hi"])
    return [(int(round(math.exp(lo + (hi - lo) * (i + 0.5) / n))), (126, 630)[i % 2], (0.5, 0.1)[i % 2],
             seed * 100 + i) for i in range(n)]


class _Cluster:
    """A jittered fcc sphere with its H, and spectral bounds found in plain torch."""

    def __init__(self, n, seed):
        self.pos = _fcc(n, seed)
        self.a, self.b = _pairs(self.pos, CUTOFF)
        self.blocks = _sk_H(self.pos, self.a, self.b)
        self.emin, self.emax = _bounds(_Op(n, self.a, self.b, self.blocks))


def _solver(case, seed):
    class Work:
        """What Solver asks of a workload."""
        positions, box, cutoff = np.zeros((case["atoms"], 3)), None, CUTOFF
        n_orb, n_atoms, mixed, jackson, order = 9, case["atoms"], True, False, case["order"]
        kT, n_electrons, n_probes, probe_seed = case["kT"], 11.0 * case["atoms"], case["probes"], seed + 52640
        sk_V = SK_V
    return api.Solver(Work())


def _fermi_moments(case, seed):
    """Moments of a sampled spectrum on [-10, 12] eV (a d band below a broad sp band), 11 electrons per
    nine states."""
    g = torch.Generator(device=DEV).manual_seed(seed)
    n = case["states"]
    e = torch.cat([torch.randn(5 * n // 9, dtype=torch.float64, device=DEV, generator=g) * 1.2 - 1.0,
                   torch.rand(n - 5 * n // 9, dtype=torch.float64, device=DEV, generator=g) * 20.0 - 9.0])
    t = torch.acos(((e.clamp(-9.8, 11.8) + 10.0) / 11.0 - 1.0))
    k = torch.arange(case["order"], dtype=torch.float64, device=DEV)
    mom = torch.cat([torch.cos(kk[:, None] * t[None]).sum(1) for kk in k.split(64)])
    return mom


def prepare(case, seed):
    kind = case["kind"]
    st = {"case": case, "seed": seed, "ctx": api.Context()}
    ctx = st["ctx"]
    if kind == "solver":
        st["solver"], st["pos"] = _solver(case, seed), _fcc(case["atoms"], seed)
    elif kind == "setup":
        st["model"], st["pos"] = _sk_model(), _fcc(case["atoms"], seed)
    elif kind == "fermi":
        st["mom"] = _fermi_moments(case, seed)
    elif kind == "sc":
        size = case["L"]
        disp = np.array([[1, 0, 0], [-1, 0, 0], [0, 1, 0], [0, -1, 0], [0, 0, 1], [0, 0, -1]], float)
        ons = torch.as_tensor(_sc_onsite(size, seed)[:, None], device=DEV)
        model = api.Model(L.TBK_MODEL_TABLE, 1, disp=disp, blocks=np.full((6, 1, 1), -1.0), onsite_site=ons)
        st["pos"] = torch.as_tensor(_cubic(size), device=DEV)
        g = api.build_neighbors(ctx, st["pos"], 1.0)
        st["model"], st["H"], st["bounds"] = model, api.assemble_H(ctx, model, st["pos"], g), (-6.6, 6.6)
    elif kind == "lattice":
        size = case["L"]
        disp, blocks = _lattice_model(seed)
        st["model"] = model = api.Model(L.TBK_MODEL_TABLE, 9, disp=disp, blocks=blocks)
        st["pos"] = torch.as_tensor(_cubic(size), device=DEV)
        g = api.build_neighbors(ctx, st["pos"], 1.5, [float(size)] * 3)
        st["H"] = api.assemble_H(ctx, model, st["pos"], g, [float(size)] * 3)
        st["bounds"] = _lattice_bounds(seed)
    elif kind == "batch":
        st["model"], st["clusters"] = _sk_model(), []
        for n, p, kT, sd in _batch(case, seed):
            c = _Cluster(n, sd)
            g = api.build_neighbors(ctx, c.pos, CUTOFF)
            st["clusters"].append((c.pos, api.assemble_H(ctx, st["model"], c.pos, g), c.emin, c.emax, sd, p,
                                   11.0 * n, kT))
    else:  # forces, direct, local: one cluster with its H and bounds
        c = _Cluster(case["atoms"], seed)
        st["model"], st["pos"], st["bounds"] = _sk_model(), c.pos, (c.emin, c.emax)
        g = api.build_neighbors(ctx, c.pos, CUTOFF)
        st["H"] = api.assemble_H(ctx, st["model"], c.pos, g)
    return st


def run(st):
    case, ctx, seed = st["case"], st["ctx"], st["seed"]
    kind = case["kind"]
    if kind == "solver":
        r = st["solver"].energies_and_forces(st["pos"])
        return {"bounds": (r.emin, r.emax), "obs": (r.mu, r.Omega, r.E, r.N), "moments": r.moments,
                "forces": r.forces}
    if kind == "setup":
        g = api.build_neighbors(ctx, st["pos"], CUTOFF)
        H = api.assemble_H(ctx, st["model"], st["pos"], g)
        return {"row_ptr": g.row_ptr, "col": g.col, "H": H.val, "bounds": api.spectral_bounds(ctx, H)}
    if kind == "fermi":
        return api.fermi_level(ctx, st["mom"], -10.0, 12.0, 11.0 * case["states"] / 9.0, case["kT"])
    if kind == "sc":
        lo, hi = st["bounds"]
        mom = api.chebyshev_moments(ctx, st["H"], lo, hi, seed, case["probes"], case["order"], fp64=True)
        return {"moments": mom, "obs": api.fermi_level(ctx, mom, lo, hi, float(case["L"] ** 3), 0.1, jackson=True)}
    if kind == "lattice":
        lo, hi = st["bounds"]
        return api.chebyshev_moments(ctx, st["H"], lo, hi, seed, case["probes"], case["order"])
    if kind == "batch":
        pos, Hs, lo, hi, sd, p, ne, kT = zip(*st["clusters"])
        mom, obs, G, F = api.batched_energies_and_forces(ctx, list(Hs), st["model"], list(pos), lo, hi, sd,
                                                         case["probes"], p, ne, kT, windowed=case["windowed"])
        return {"moments": mom, "obs": obs, "forces": F}
    lo, hi = st["bounds"]
    if kind == "forces":
        mom, obs, G, F = api.energies_and_forces(ctx, st["H"], st["model"], st["pos"], None, lo, hi, seed,
                                                 case["probes"], case["order"], 11.0 * case["atoms"], case["kT"],
                                                 fp64=case["fp64"], want_G=True)
        return {"moments": mom, "obs": obs, "G": G, "forces": F}
    if kind == "direct":
        P, Q, _ = api.direct_density(ctx, st["H"], None, None, None, lo, hi, seed, case["probes"], case["order"],
                                     6.0, case["kT"])
        return {"P": P, "Q": Q}
    P, Q = api.local_density(ctx, st["H"], st["pos"], None, case["r_max"], lo, hi, case["order"], 6.0, case["kT"])
    return {"P": P, "Q": Q}


# ---- what a pass cannot do without -----------------------------------------------------------------

def _fcc_count(n, r_max):
    """Pairs within r_max (self included) of the n-site sphere without jitter."""
    s = _fcc_sites(n)
    r = int(np.abs(s).max())
    w = int(math.ceil(r_max / (FCC_A / 2.0))) + 1
    grid = np.zeros((2 * (r + w) + 1,) * 3, dtype=bool)
    c = s + r + w
    grid[c[:, 0], c[:, 1], c[:, 2]] = True
    total = 0
    for o in np.stack(np.meshgrid(*[np.arange(-w, w + 1)] * 3, indexing="ij"), -1).reshape(-1, 3):
        if o.sum() % 2 == 0 and (o * o).sum() <= (r_max / (FCC_A / 2.0)) ** 2:
            total += int(grid[c[:, 0] + o[0], c[:, 1] + o[1], c[:, 2] + o[2]].sum())
    return total


def work(case):
    kind = case["kind"]
    if kind == "fermi":
        return {"bytes": 8.0 * case["order"], "flops": 4.0 * case["order"] * 4 * case["order"]}
    if kind == "sc":
        n, s, p = case["L"] ** 3, case["probes"], case["order"]
        return {"bytes": 8.0 * (7 * n + p), "flops": 2.0 * 7 * n * s * (p // 2)}
    if kind == "lattice":
        n, s, p = case["L"] ** 3, case["probes"], case["order"]
        return {"bytes": 8.0 * (19 * 81 * n + p), "flops": 2.0 * 81 * 19 * n * s * (p // 2)}
    if kind == "setup":
        nnz = _fcc_count(case["atoms"], CUTOFF)
        return {"bytes": 24.0 * case["atoms"] + nnz * (648.0 + 4.0), "flops": nnz * (400.0 + 64 * 2 * 81)}
    if kind == "batch":
        by = fl = 0.0
        for n, p, _, _ in _batch(case, 0):
            nnz = _fcc_count(n, CUTOFF)
            by += nnz * 648.0 + 48.0 * n
            fl += 3 * 2.0 * 81 * nnz * case["probes"] * (p // 2)
        return {"bytes": by, "flops": fl}
    n = case["atoms"]
    nnz = _fcc_count(n, CUTOFF)
    if kind == "local":
        regions = _fcc_count(n, case["r_max"])
        # the blocks inside the regions: about the mean row of H for the atoms of each region
        return {"bytes": nnz * 648.0 * 3, "flops": 2.0 * 81 * 9 * regions * 0.75 * nnz / n * case["order"]}
    p, s = case["order"], case["probes"]
    if kind == "direct":
        return {"bytes": nnz * 648.0 * 3, "flops": 2.0 * 81 * nnz * s * (p + 2)}
    # solver, forces: K = p/2 block products forward, as many backward, as many outer products
    return {"bytes": nnz * 648.0 * 2 + 48.0 * n, "flops": 3 * 2.0 * 81 * nnz * s * (p // 2)}


# ---- the same quantities in plain torch, 64 bits ------------------------------------------------------

def _pairs(pos, cutoff, box=None):
    """All (a, b) with |r_b - r_a| <= cutoff, a-major, ascending."""
    a, b = [], []
    for i0 in range(0, pos.shape[0], 1024):
        d = pos[None] - pos[i0:i0 + 1024, None]
        if box is not None:
            d = d - box * torch.round(d / box)
        i, j = torch.nonzero((d * d).sum(-1) <= cutoff * cutoff, as_tuple=True)
        a.append(i + i0)
        b.append(j)
    return torch.cat(a), torch.cat(b)


def _d_tensors():
    """The d orbitals dxy, dyz, dzx, dx2-y2, d3z2-r2 as quadratic forms u^T Q u on the unit sphere."""
    q = torch.zeros(5, 3, 3, dtype=torch.float64, device=DEV)
    h = math.sqrt(3.0) / 2.0
    for i, (x, y) in enumerate(((0, 1), (1, 2), (2, 0))):
        q[i, x, y] = q[i, y, x] = h
    q[3, 0, 0], q[3, 1, 1] = h, -h
    q[4] = torch.diag(torch.tensor([-0.5, -0.5, 1.0], dtype=torch.float64, device=DEV))
    return q


def _sk_blocks(d):
    """Two-centre Slater-Koster blocks for bond vectors d (m, 3) -> (m, 9, 9)."""
    r = d.norm(dim=1, keepdim=True)
    u = d / r
    sss, sps, sds, pps, ppp, pds, pdp, dds, ddp, ddd = (torch.exp(-DECAY * (r / R0 - 1.0)) * v for v in SK_V)
    Q = _d_tensors()
    Qu = torch.einsum("ixy,my->mix", Q, u)               # Q_i u
    S = torch.einsum("mix,mx->mi", Qu, u)                # u^T Q_i u
    I3, I5 = torch.eye(3, dtype=torch.float64, device=DEV), torch.eye(5, dtype=torch.float64, device=DEV)
    uu, SS = u[:, :, None] * u[:, None, :], S[:, :, None] * S[:, None, :]
    pi = (4.0 / 3.0) * (torch.einsum("mix,mjx->mij", Qu, Qu) - SS)
    e = lambda v: v[:, :, None]
    pp = uu * e(pps) + (I3 - uu) * e(ppp)
    uS = u[:, :, None] * S[:, None, :]
    pd = uS * e(pds) + (2.0 / math.sqrt(3.0)) * (Qu.transpose(1, 2) - uS) * e(pdp)
    dd = SS * e(dds) + pi * e(ddp) + (I5 - SS - pi) * e(ddd)
    sp, sd = (u * sps)[:, None], (S * sds)[:, None]
    top = torch.cat([e(sss), sp, sd], 2)
    mid = torch.cat([-sp.transpose(1, 2), pp, pd], 2)
    low = torch.cat([sd.transpose(1, 2), -pd.transpose(1, 2), dd], 2)
    return torch.cat([top, mid, low], 1)


def _sk_H(pos, a, b):
    off = a != b
    out = torch.diag(torch.tensor([ONSITE[0]] + [ONSITE[1]] * 3 + [ONSITE[2]] * 5, dtype=torch.float64,
                                  device=DEV)).repeat(len(a), 1, 1)
    return out.index_put((torch.nonzero(off)[:, 0],), _sk_blocks(pos[b[off]] - pos[a[off]]))


class _Op:
    """Block-sparse operator as a padded neighbour table: y -> scale (H - shift) y."""

    def __init__(self, n, a, b, blocks, shift=0.0, scale=1.0):
        B = blocks.shape[1]
        count = torch.bincount(a, minlength=n)
        slot = torch.arange(len(a), device=DEV) - (count.cumsum(0) - count)[a]
        m = int(count.max())
        self.n, self.B, self.m, self.a, self.b, self.scale = n, B, m, a, b, scale
        self.cols = torch.zeros(n, m, dtype=torch.int64, device=DEV)
        self.cols[a, slot] = b
        h = torch.zeros(n, m, B, B, dtype=torch.float64, device=DEV)
        h[a, slot] = blocks
        own = torch.nonzero(a == b)[:, 0]
        h[a[own], slot[own]] -= shift * torch.eye(B, dtype=torch.float64, device=DEV)
        self.h = (h * scale).permute(0, 2, 1, 3).reshape(n, B, m * B).contiguous()

    def __call__(self, y):
        y3 = y.view(self.n, self.B, -1)
        out = torch.empty_like(y3)
        step = max(1, int(2e8 // (self.m * self.B * y3.shape[2])))
        for i in range(0, self.n, step):
            c = self.cols[i:i + step]
            x = y3[c.reshape(-1)].view(c.shape[0], self.m * self.B, -1)
            torch.bmm(self.h[i:i + step], x, out=out[i:i + step])
        return out.view(y.shape)

    def outer(self, y, x):
        """sum over columns of y[row block a] x[row block b]^T on every stored block."""
        y3, x3 = y.view(self.n, self.B, -1), x.view(self.n, self.B, -1)
        out = torch.empty(len(self.a), self.B, self.B, dtype=torch.float64, device=DEV)
        step = max(1, int(1e8 // (self.B * y3.shape[2])))
        for i in range(0, len(self.a), step):
            torch.bmm(y3[self.a[i:i + step]], x3[self.b[i:i + step]].transpose(1, 2), out=out[i:i + step])
        return out


def _mapped(n, a, b, blocks, lo, hi):
    return _Op(n, a, b, blocks, 0.5 * (lo + hi), 2.0 / (hi - lo))


def _shift_right(z, k):
    return (z >> k) & ((1 << (64 - k)) - 1)


def _signed(v):
    v &= M64
    return v - (1 << 64) if v >> 63 else v


def _probes(rows, s, seed):
    """Rademacher probes: the top bit of SplitMix64 output number row 2^32 + probe + 1."""
    i = (torch.arange(rows, device=DEV)[:, None] << 32) + torch.arange(s, device=DEV)[None] + 1
    z = i * _signed(0x9E3779B97F4A7C15) + _signed(seed)
    z = (z ^ _shift_right(z, 30)) * _signed(0xBF58476D1CE4E5B9)
    z = (z ^ _shift_right(z, 27)) * _signed(0x94D049BB133111EB)
    return torch.where(z ^ _shift_right(z, 31) < 0, -1.0, 1.0).to(torch.float64)


def _bounds(op, steps=64, margin=0.01):
    """Extreme Ritz values of a plain Lanczos run with their residuals, widened by the margin."""
    n = op.n * op.B
    v = _probes(n, 1, BOUNDS_SEED) / math.sqrt(n)
    prev, beta, al, be = torch.zeros_like(v), 0.0, [], []
    for _ in range(min(steps, n)):
        w = op(v) - beta * prev
        al.append(float((w * v).sum()))
        w = w - al[-1] * v
        beta = float(w.norm())
        be.append(beta)
        prev, v = v, w / beta
    T = np.diag(al) + np.diag(be[:-1], 1) + np.diag(be[:-1], -1)
    th, z = np.linalg.eigh(T)
    lo, hi = th[0] - be[-1] * abs(z[-1, 0]), th[-1] + be[-1] * abs(z[-1, -1])
    return lo - margin * (hi - lo), hi + margin * (hi - lo)


def _lattice_bounds(seed):
    """Bounds of the lattice band from H(k) on a 24^3 grid, widened by 1 %."""
    disp, blocks = _lattice_model(seed)
    k = torch.as_tensor(_cubic(24) * (2 * math.pi / 24), device=DEV)
    ph = torch.exp(1j * (k @ torch.as_tensor(disp, device=DEV).T))
    H = torch.einsum("kd,dij->kij", ph, torch.as_tensor(blocks, device=DEV).to(torch.complex128))
    H = torch.cat([H.real, -H.imag], 2), torch.cat([H.imag, H.real], 2)
    e = np.linalg.eigvalsh(torch.cat(H, 1)[::7].cpu().numpy())
    w = e.max() - e.min()
    return float(e.min() - 0.02 * w), float(e.max() + 0.02 * w)


def _panels(op, R, p):
    ys = [R, op(R)]
    for _ in range(2, p // 2 + 1):
        ys.append(2.0 * op(ys[-1]) - ys[-2])
    return ys


def _moments_of(op, R, p, ys=None):
    """mu_0 .. mu_{p-1} through C_m C_n = (C_{m+n} + C_{|m-n|})/2."""
    s = R.shape[1]
    mom = torch.zeros(p + 2, dtype=torch.float64, device=DEV)
    y0, y1 = R, op(R)
    m1 = (y1 * y0).sum() / s
    mom[0], mom[1] = R.shape[0], m1
    for k in range(1, p // 2 + 1):
        if k > 1:
            y0, y1 = y1, (ys[k] if ys else 2.0 * op(y1) - y0)
            mom[2 * k - 1] = 2.0 * (y1 * y0).sum() / s - m1
        mom[2 * k] = 2.0 * (y1 * y1).sum() / s - R.shape[0]
    return mom[:p]


def _jackson(p):
    k, q = torch.arange(p, dtype=torch.float64, device=DEV), math.pi / (p + 1)
    return ((p - k + 1) * torch.cos(q * k) + torch.sin(q * k) / math.tan(q)) / (p + 1)


def _nodes(p, lo, hi):
    m = max(4 * p, 256)
    t = math.pi * (torch.arange(m, dtype=torch.float64, device=DEV) + 0.5) / m
    x = torch.cos(t)
    return t, lo * (1 - x) / 2 + hi * (1 + x) / 2


def _occupation(e, mu, kT):
    return 2.0 * torch.sigmoid(-(e - mu) / kT)


def _free(e, mu, kT):
    return -2.0 * kT * torch.nn.functional.softplus(-(e - mu) / kT, threshold=1000.0)


def _observables(mom, lo, hi, n_e, kT, damp=None):
    p = len(mom)
    t, e = _nodes(p, lo, hi)
    w = mom * (1.0 if damp is None else damp)
    w = torch.cat([w[:1], 2.0 * w[1:]])
    k = torch.arange(p, dtype=torch.float64, device=DEV)
    rho = torch.cat([torch.cos(tt[:, None] * k[None]) @ w for tt in t.split(1024)]) / len(t)
    x0, x1 = lo, hi
    for _ in range(200):
        mid = 0.5 * (x0 + x1)
        if float((_occupation(e, mid, kT) * rho).sum()) < n_e:
            x0 = mid
        else:
            x1 = mid
        if x1 - x0 < 1e-13 * (hi - lo):
            break
    mu = 0.5 * (x0 + x1)
    f = _occupation(e, mu, kT)
    return mu, float((_free(e, mu, kT) * rho).sum()), float((e * f * rho).sum()), float((f * rho).sum())


def _coefficients(fn, p, lo, hi, mu, kT):
    t, e = _nodes(p, lo, hi)
    h = fn(e, mu, kT)
    k = torch.arange(p, dtype=torch.float64, device=DEV)
    c = torch.cat([torch.cos(kk[:, None] * t[None]) @ h for kk in k.split(512)]) * (2.0 / len(t))
    c[0] *= 0.5
    return c.tolist()


def _density(op, ys, p, c, half_width):
    """dOmega/dH on the pattern: reverse mode through the doubled moments, symmetrised."""
    s, K = ys[0].shape[1], p // 2
    w, v = [0.0] * (K + 2), [0.0] * (K + 2)
    for k in range(1, K + 1):
        w[k] = 2.0 * c[2 * k] if 2 * k < p else 0.0
        v[k] = 2.0 * c[2 * k - 1] if k >= 2 and 2 * k - 1 < p else 0.0
    v[1] = c[1] - sum(c[3:p:2])
    G = torch.zeros(len(op.a), op.B, op.B, dtype=torch.float64, device=DEV)
    b1 = b2 = None                                        # ybar_{k+1}, ybar_{k+2}
    for k in range(K, -1, -1):
        if b1 is not None:
            G += op.outer(ys[k], b1) * (2.0 if k else 1.0)
        if k:
            g = (2.0 * w[k] * ys[k] + v[k] * ys[k - 1]) / s
            if k < K:
                g += v[k + 1] / s * ys[k + 1] + 2.0 * op(b1)
            if b2 is not None:
                g -= b2
            b1, b2 = g, b1
    key = op.a * op.n + op.b
    tr = torch.searchsorted(key, op.b * op.n + op.a)
    return 0.5 * (G + G[tr].transpose(1, 2)) / half_width


def _forces(pos, a, b, G):
    x = pos.clone().requires_grad_(True)
    (_sk_H(x, a, b) * G).sum().backward()
    return -x.grad


def _energies_and_forces(c, lo, hi, seed, s, p, n_e, kT):
    n = c.pos.shape[0]
    op = _mapped(n, c.a, c.b, c.blocks, lo, hi)
    R = _probes(9 * n, s, seed)
    ys = _panels(op, R, p)
    mom = _moments_of(op, R, p, ys)
    obs = _observables(mom, lo, hi, n_e, kT)
    G = _density(op, ys, p, _coefficients(_free, p, lo, hi, obs[0], kT), 0.5 * (hi - lo))
    return mom, obs, G, _forces(c.pos, c.a, c.b, G)


def _polynomial(apply, E, c):
    """sum_k c_k C_k(H^) E by the three-term recurrence."""
    y0, y1 = E, apply(E)
    X = c[0] * y0 + c[1] * y1
    for k in range(2, len(c)):
        y0, y1 = y1, 2.0 * apply(y1) - y0
        X = X + c[k] * y1
    return X


def _local(case, c):
    """Every atom's region as a dense local problem, in batches of atoms."""
    n = c.pos.shape[0]
    coef = _coefficients(_occupation, case["order"], c.emin, c.emax, 6.0, case["kT"])
    dense = torch.zeros(n, n, 9, 9, dtype=torch.float64, device=DEV)
    dense[c.a, c.b] = c.blocks
    ra, rb = _pairs(c.pos, case["r_max"])
    count = torch.bincount(ra, minlength=n)
    m = int(count.max())
    slot = torch.arange(len(ra), device=DEV) - (count.cumsum(0) - count)[ra]
    region = torch.full((n, m), -1, dtype=torch.int64, device=DEV)
    region[ra, slot] = rb
    P, Q = torch.zeros(n, n, 9, 9, dtype=torch.float64, device=DEV), torch.zeros(n, n, 9, 9, dtype=torch.float64,
                                                                                device=DEV)
    shift, scale = 0.5 * (c.emin + c.emax), 2.0 / (c.emax - c.emin)
    for i in range(0, n, 64):
        g = region[i:i + 64]
        live = (g >= 0).to(torch.float64)
        gg = g.clamp(min=0)
        q = g.shape[0]
        H = dense[gg[:, :, None], gg[:, None, :]] * (live[:, :, None] * live[:, None, :])[..., None, None]
        H = H.permute(0, 1, 3, 2, 4).reshape(q, 9 * m, 9 * m)
        own = torch.nonzero(g == torch.arange(i, i + q, device=DEV)[:, None])[:, 1]
        E = torch.zeros(q, m, 9, 9, dtype=torch.float64, device=DEV)
        E[torch.arange(q, device=DEV), own] = torch.eye(9, dtype=torch.float64, device=DEV)
        X = _polynomial(lambda y: scale * (torch.bmm(H, y) - shift * y), E.view(q, 9 * m, 9), coef)
        for out, Y in ((P, X), (Q, torch.bmm(H, X))):
            at = torch.nonzero(g >= 0, as_tuple=True)
            out[g[at], i + at[0]] = Y.view(q, m, 9, 9)[at]
    return {"P": P[c.a, c.b], "Q": Q[c.a, c.b]}


def _sc_onsite(size, seed):
    return np.random.default_rng(seed).uniform(-0.5, 0.5, size=size ** 3)


def exact(case, seed):
    kind = case["kind"]
    if kind == "fermi":
        return _observables(_fermi_moments(case, seed), -10.0, 12.0, 11.0 * case["states"] / 9.0, case["kT"])
    if kind == "sc":
        pos = torch.as_tensor(_cubic(case["L"]), device=DEV)
        a, b = _pairs(pos, 1.0)
        val = torch.where(a == b, torch.as_tensor(_sc_onsite(case["L"], seed), device=DEV)[a], -1.0)[:, None, None]
        R = _probes(len(pos), case["probes"], seed)
        mom = _moments_of(_mapped(len(pos), a, b, val, -6.6, 6.6), R, case["order"])
        return {"moments": mom, "obs": _observables(mom, -6.6, 6.6, float(len(pos)), 0.1, _jackson(case["order"]))}
    if kind == "lattice":
        pos, size = torch.as_tensor(_cubic(case["L"]), device=DEV), case["L"]
        disp, blocks = _lattice_model(seed)
        a, b = _pairs(pos, 1.5, float(size))
        d = pos[b] - pos[a]
        d = torch.round(d - size * torch.round(d / size)).long() + 1
        table = torch.zeros(27, 9, 9, dtype=torch.float64, device=DEV)
        at = torch.as_tensor(disp, device=DEV).long() + 1
        table[at[:, 0] * 9 + at[:, 1] * 3 + at[:, 2]] = torch.as_tensor(blocks, device=DEV)
        op = _mapped(len(pos), a, b, table[d[:, 0] * 9 + d[:, 1] * 3 + d[:, 2]], *_lattice_bounds(seed))
        return _moments_of(op, _probes(9 * len(pos), case["probes"], seed), case["order"])
    if kind == "batch":
        mom, obs, F = [], [], []
        for n, p, kT, sd in _batch(case, seed):
            c = _Cluster(n, sd)
            m, o, _, f = _energies_and_forces(c, c.emin, c.emax, sd, case["probes"], p, 11.0 * n, kT)
            mom.append(m)
            obs.append(o)
            F.append(f)
        return {"moments": mom, "obs": np.array(obs), "forces": F}
    c = _Cluster(case["atoms"], seed)
    lo, hi = c.emin, c.emax
    if kind == "setup":
        row = torch.cat([torch.zeros(1, dtype=torch.int64, device=DEV), torch.bincount(c.a).cumsum(0)])
        return {"row_ptr": row.int(), "col": c.b.int(), "H": c.blocks, "bounds": (lo, hi)}
    if kind == "solver":
        mom, obs, _, F = _energies_and_forces(c, lo, hi, seed + 52640, case["probes"], case["order"],
                                              11.0 * case["atoms"], case["kT"])
        return {"bounds": (lo, hi), "obs": obs, "moments": mom, "forces": F}
    if kind == "forces":
        mom, obs, G, F = _energies_and_forces(c, lo, hi, seed, case["probes"], case["order"], 11.0 * case["atoms"],
                                              case["kT"])
        return {"moments": mom, "obs": obs, "G": G, "forces": F}
    if kind == "local":
        return _local(case, c)
    n, s = case["atoms"], case["probes"]
    R = _probes(9 * n, s, seed)
    X = _polynomial(_mapped(n, c.a, c.b, c.blocks, lo, hi), R,
                    _coefficients(_occupation, case["order"], lo, hi, 6.0, case["kT"]))
    H = _Op(n, c.a, c.b, c.blocks)
    return {"P": H.outer(X, R) / s, "Q": H.outer(H(X), R) / s}
