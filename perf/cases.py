"""Performance cases of the LDPM library: what its users run, through its public entry points.

A specimen here is a prism of nx * ny * nz copies of one periodic Delaunay block of `block` particles
(about 6.7 tetrahedra per particle, valences spread as in a random packing, a free jagged surface), at
the particle density and the diameters (2 to 4 mm) of the repository's 50 mm tension cube.  Repeating a
block keeps the mesh generation of the largest specimens to a second or two; the library sees an
ordinary specimen.  A case has one of these kinds:

  steps    `steps` time steps from a restart state, then the whole state read out on the device
  log      `steps` times one time step and an energy / reaction read-back (a load-displacement curve)
  batch    `steps` time steps of `batch` specimens of uneven size from rest under an initial velocity
  adjoint  objective and gradient with respect to every facet's E0, alpha and sigma_t over `steps` steps

The restart state is strained as in the middle of a test: `tension` stretches a band past the tensile
limit (softening facets, the rest elastic, tension and compression branches mixed), `compression` is a
confined compression up to the compressive yield limit, `elastic` is free vibration with linear
facets.  Mixed-precision outputs are kept in single precision, the precision of the facet stage that
makes them; FP64 outputs in double.
"""
from __future__ import annotations

import functools
import math
import types

import numpy as np
import torch

from paper_2603_13190_gb300 import ldpm, specimen, workloads

SPACING = 50.0 / 25000 ** (1.0 / 3.0)  # mm per particle of the 50 mm tension cube
RAMP = 4e-4                            # s, ramp of the prescribed velocities; restart states are past it
L2_BYTES = 126e6
SLOT_A = [a for a, _ in specimen.TET_EDGES for _ in (0, 1)]
SLOT_B = [b for _, b in specimen.TET_EDGES for _ in (0, 1)]


def _case(kind, precision, loading, block, nx, ny, nz, steps, hetero=False, batch=1, ckpt=0):
    return dict(kind=kind, precision=precision, loading=loading, block=block, nx=nx, ny=ny, nz=nz, steps=steps,
                hetero=hetero, batch=batch, ckpt=ckpt)


def listed():
    return [
        # the paper's smallest test (free vibration, 18k facets, Sec. 4.1), double precision: launch latency
        {"name": "vibration_fp64_small"} | _case("steps", "fp64", "elastic", 331, 1, 1, 1, 64),
        # a 25 mm dog-bone neck, the size of a quick tensile study
        {"name": "tension_mixed_small"} | _case("steps", "mixed", "tension", 523, 2, 1, 3, 32),
        # the 50 mm tension cube (1.8M facets) in the middle of a run
        {"name": "tension_mixed"} | _case("steps", "mixed", "tension", 997, 3, 3, 3, 20),
        # tensile fracture in double precision, as the paper's solvers run it
        {"name": "tension_fp64"} | _case("steps", "fp64", "tension", 811, 2, 2, 3, 10),
        # confined compression in double precision
        {"name": "compression_fp64"} | _case("steps", "fp64", "compression", 901, 2, 3, 3, 10),
        # the 100 mm confined-compression cube, the largest single specimen
        {"name": "compression_mixed_large"} | _case("steps", "mixed", "compression", 1013, 5, 5, 6, 10),
        # per-facet material (spatial variability of strength and stiffness)
        {"name": "tension_mixed_hetero"} | _case("steps", "mixed", "tension", 607, 2, 2, 2, 24, hetero=True),
        # load-displacement curve: energies and reactions after every step
        {"name": "log_mixed"} | _case("log", "mixed", "tension", 467, 2, 2, 2, 24),
        # random realisations of uneven size stepped together (Sec. 4.5, unconfined compression)
        {"name": "batch_mixed"} | _case("batch", "mixed", "compression", 389, 3, 3, 4, 16, batch=12),
        # sensitivities for calibration: mixed precision on a mid-size specimen, checkpointed
        {"name": "adjoint_mixed"} | _case("adjoint", "mixed", "pretension", 701, 3, 3, 3, 400, ckpt=100),
        # and a small specimen in double precision
        {"name": "adjoint_fp64_small"} | _case("adjoint", "fp64", "pretension", 449, 1, 1, 2, 48, ckpt=12),
    ]


def draw(rng):
    kind = rng.choice(["steps", "steps", "steps", "log", "batch", "adjoint"])
    precision = rng.choice(["mixed", "mixed", "fp64"])
    loading = {"adjoint": "pretension", "batch": "compression"}.get(kind)
    loading = loading or rng.choice(["tension", "compression", "elastic"])
    top = {"steps": 80000, "log": 20000, "batch": 12000, "adjoint": 20000}[kind] // (1 if precision == "mixed" else 5)
    want = math.exp(rng.uniform(math.log(300), math.log(top)))  # particles
    n = [max(1, round(rng.uniform(0.7, 1.4) * (want / 800) ** (1 / 3))) for _ in range(3)]
    block = min(1200, max(230, round(want / (n[0] * n[1] * n[2]))))
    steps = rng.randint(24, 64) if kind == "adjoint" else rng.randint(4, 32)
    return _case(kind, precision, loading, block, *n, steps,
                 hetero=kind in ("steps", "adjoint") and rng.random() < 0.25,
                 batch=rng.randint(2, 8) if kind == "batch" else 1,
                 ckpt=rng.randint(7, 40) if kind == "adjoint" else 0)


# --------------------------------------------------------------------------------------------------
# Inputs.
# --------------------------------------------------------------------------------------------------
@functools.lru_cache(maxsize=4)
def _block(n):
    """Periodic Delaunay mesh of n points in the unit cube: points, tetrahedra, the vertices' images.  It
    depends on n alone, so that a case has the same sizes for every seed; the seed moves the points."""
    rng = np.random.default_rng(n)
    g = math.ceil(n ** (1.0 / 3.0))
    cell = np.sort(rng.permutation(g ** 3)[:n])
    p = (np.stack(np.unravel_index(cell, (g, g, g)), 1) + rng.uniform(0.12, 0.88, (n, 3))) / g
    s = np.stack(np.meshgrid(*[(-1, 0, 1)] * 3, indexing="ij"), -1).reshape(-1, 3)
    img = (p[None] + s[:, None]).reshape(-1, 3)
    near = np.nonzero(np.all((img > -0.55) & (img < 1.55), axis=1))[0]
    tri = specimen.Delaunay(img[near]).simplices
    corner = img[near][tri]
    mid = corner.mean(1)
    d = corner[:, 1:] - corner[:, :1]
    vol = np.abs(np.linalg.det(d))
    keep = np.all((mid >= 0) & (mid < 1), axis=1) & (vol > 1e-6 * np.median(vol))
    ids = near[tri[keep]]
    return p, ids % n, s[ids // n]


def _specimen(case, seed, counts):
    """The prism of counts[0] x counts[1] x counts[2] blocks as a specimen.Specimen."""
    n = case["block"]
    p, ids, img = _block(n)
    m = np.asarray(counts)
    rng = np.random.default_rng(seed + 1)
    p = p + rng.uniform(-0.03, 0.03, p.shape) / n ** (1.0 / 3.0)
    size = SPACING * n ** (1.0 / 3.0)
    diameter = specimen.fuller_diameters(n, 2.0, 4.0, 0.4, rng)[rng.permutation(n)]
    corner = ((p[ids] + img) * size).reshape(-1, 3)
    vtx = specimen.tessellate(corner, 0.2 * diameter[ids].reshape(-1), np.arange(4 * len(ids)).reshape(-1, 4))[3]
    vtx = vtx.reshape(len(ids), 12, 3, 3)
    tile = np.stack(np.meshgrid(*[np.arange(k) for k in m], indexing="ij"), -1).reshape(-1, 3)
    tets, verts = [], []
    for t in tile:
        w = t + img
        ok = np.all((w >= 0) & (w < m), axis=(1, 2))
        tets.append(((w[ok, :, 0] * m[1] + w[ok, :, 1]) * m[2] + w[ok, :, 2]) * n + ids[ok])
        verts.append(vtx[ok] + t * size)
    tets = np.concatenate(tets)
    x = ((p[None] + tile[:, None]) * size).reshape(-1, 3)
    used = np.zeros(len(x), bool)
    used[tets.reshape(-1)] = True
    tets = (np.cumsum(used) - 1)[tets].astype(np.int32)
    return specimen.Specimen(
        x=np.ascontiguousarray(x[used]), diameter=np.tile(diameter, len(tile))[used], tets=tets,
        facet_pi=tets[:, SLOT_A].reshape(-1), facet_pj=tets[:, SLOT_B].reshape(-1),
        facet_tet=np.repeat(np.arange(len(tets), dtype=np.int32), 12),
        facet_vtx=np.concatenate(verts).reshape(-1, 9), edge=float(size * m[2]), d_min=2.0, d_max=4.0)


def _counts(case, k):
    """Blocks of specimen k: batches have uneven ones."""
    full = [case["nx"], case["ny"], case["nz"]]
    if case["kind"] != "batch":
        return full
    return [max(1, c - (k * (2 * i + 3)) % 3) for i, c in enumerate(full)]


def _build(case, seed, k=0):
    """Specimen k of a case with its material, boundary conditions, time step and restart state; the
    reference formulation of it (tensors on the device); per-facet parameters or None."""
    seed = 1000 * seed + 10 * k
    spec = _specimen(case, seed, _counts(case, k))
    mat = dict(workloads.WORKLOAD_MATERIAL, elastic=int(case["loading"] == "elastic"))
    rng = np.random.default_rng(seed + 2)
    x, N = spec.x, spec.n_particles
    lo, hi = x.min(0), x.max(0)
    xi = (x - lo) / (hi - lo)
    bc = workloads.free_bc(N)
    low, high = x < lo + 0.8 * SPACING, x > hi - 0.8 * SPACING
    bottom, top = low[:, 2], high[:, 2]
    limit = mat["sigma_t"] / mat["E0"] if "tension" in case["loading"] else mat["sigma_c0"] / mat["E0"]
    wave = np.cos(2 * np.pi * (xi[:, 2] + rng.uniform(0, 1)))
    L = hi[2] - lo[2]
    q, v = np.zeros((N, 6)), np.zeros((N, 6))
    if case["loading"] == "elastic":
        bc.mask[bottom] = workloads.FIXED
        v[:, 0] = 10.0 * np.sin(0.5 * np.pi * xi[:, 2]) * (1 + 0.2 * wave)
        v[bottom] = 0.0
        q[:, 0] = 1e-4 * np.sin(0.5 * np.pi * xi[:, 2])
        q[bottom] = 0.0
    elif case["loading"] == "compression":
        for ax in range(3):
            for face, sign in ((low[:, ax], 1.0), (high[:, ax], -1.0)):
                if case["kind"] == "batch" and ax < 2:
                    continue  # unconfined: platens only
                bc.mask[face, ax] = workloads.PRESCRIBED
                bc.vel[face, ax] = 25.0 * sign
        q[:, :3] = -limit * (0.6 * (x - lo) + 0.06 * (hi - lo) * np.sin(2 * np.pi * xi) * rng.uniform(0.5, 1.0, 3))
    else:
        level = 0.95 if case["loading"] == "tension" else 0.35
        for face in (bottom, top):
            bc.mask[np.ix_(face, [0, 1, 2, 3, 4])] = workloads.FIXED
        bc.mask[top, 2] = workloads.PRESCRIBED
        bc.vel[top, 2] = 50.0 if case["loading"] == "tension" else 5.0
        q[:, 2] = limit * level * (x[:, 2] - lo[2] + 0.08 * L * wave)
        q[:, :2] = -0.15 * limit * level * (x[:, :2] - 0.5 * (lo + hi)[:2])
        v[:, 2] = bc.vel[top, 2].max() * xi[:, 2]
    if case["loading"] != "elastic":
        rough = (0.005 if case["loading"] == "compression" else 0.02) * limit
        q[:, :3] += rough * SPACING * rng.standard_normal((N, 3))
        q[:, 3:] += rough * rng.standard_normal((N, 3))
    if case["kind"] == "batch":  # batches start from rest positions: an initial velocity loads them
        q[:] = 0.0
        v[:, 2] = -1000.0 * xi[:, 2] * (1 + 0.1 * rng.standard_normal(N))
        bc.ramp_time = 0.0
    else:
        bc.ramp_time = RAMP
    v[bc.mask == workloads.FIXED] = 0.0
    v = np.where(bc.mask == workloads.PRESCRIBED, bc.vel, v)
    bc.v0 = v
    par = None
    if case["hetero"]:
        F = spec.n_facets
        par = [mat[name] * np.exp(0.1 * rng.standard_normal(F)) for name in ("E0", "alpha", "sigma_t")]
    ref = _Reference(spec, mat, bc, par)
    restart = case["kind"] != "batch"
    step0 = math.ceil(RAMP / ref.dt) + 1 if restart else 0
    ref.restart(q, v, step0, strained=restart)
    return types.SimpleNamespace(spec=spec, mat=mat, bc=bc, par=par, ref=ref, q=q, v=v, step0=step0)


def prepare(case, seed):
    stream = torch.cuda.Stream()
    built = [_build(case, seed, k) for k in range(case["batch"])]
    b = built[0]
    if case["kind"] == "batch":
        model = ldpm.Batch([c.spec for c in built], [c.mat for c in built], precision=case["precision"],
                           dts=[c.ref.dt for c in built], bcs=[c.bc for c in built], stream=stream)
    else:
        model = ldpm.Model(b.spec, b.mat, precision=case["precision"], dt=b.ref.dt, bc=b.bc, stream=stream)
        if b.par is not None:
            model.set_facet_params(*b.par)
        model.set_state(b.q, b.v, b.ref.hist5().cpu().numpy(), b.step0)
    N, F = (sum(getattr(c.spec, a) for c in built) for a in ("n_particles", "n_facets"))
    out = [torch.zeros(s, dtype=torch.float64, device="cuda") for s in ((N, 6), (N, 6), (F, 5))]
    seeds = np.zeros((N, 6))
    seeds[b.bc.mask[: N] == workloads.PRESCRIBED if case["batch"] == 1 else slice(0)] = 1.0
    torch.cuda.synchronize()
    return types.SimpleNamespace(case=case, model=model, stream=stream, out=out, seeds=seeds)


def run(state):
    case, model = state.case, state.model
    if case["kind"] == "adjoint":
        J, *grads = model.adjoint(case["steps"], state.seeds, ckpt_every=case["ckpt"])
        if case["precision"] == "mixed":
            J, grads = np.float32(J), [g.astype(np.float32) for g in grads]
        return {"objective": J, "grads": grads}
    logged = {}
    if case["kind"] == "log":
        energy, reaction = np.zeros((case["steps"], 3)), np.zeros((case["steps"], 12))
        for i in range(case["steps"]):
            model.step(1)
            e, r = model.energy()
            energy[i], reaction[i] = e[:3], r
        if case["precision"] == "mixed":
            energy, reaction = energy.astype(np.float32), reaction.astype(np.float32)
        logged = {"energy": energy, "reaction": reaction}
    else:
        model.step(case["steps"])
    with torch.cuda.stream(state.stream):
        ldpm.ldpm_get_state_device(model.h, *(t.data_ptr() for t in state.out), 0)
        q, v, hist = (t.float() for t in state.out) if case["precision"] == "mixed" else state.out
    return {"q": q, "v": v, "hist": hist} | logged


# --------------------------------------------------------------------------------------------------
# Work.
# --------------------------------------------------------------------------------------------------
def work(case):
    """Per step and facet: geometry read (4 values), history read and written (8 values); per
    tetrahedron its 4 vertex ids; per particle q, v, force and energy sums read and written, position and
    constants read.  A working set that fits L2 passes through memory once per call."""
    R = 4 if case["precision"] == "mixed" else 8
    _, _, img = _block(case["block"])
    span = img.max(1) - img.min(1)
    N = T = 0
    for k in range(case["batch"]):
        m = np.asarray(_counts(case, k))
        N += case["block"] * int(np.prod(m))
        T += int(np.prod(np.maximum(m - span, 0), axis=1).sum())
    F = 12 * T
    once = F * 12 * R + 16 * T + N * (2 * 14 + 9) * 8
    sweeps = case["steps"] if once > L2_BYTES else 1
    flops = F * (190 if case["loading"] != "elastic" else 140) + N * 60
    read_out = 8 * (12 * N + 5 * F)
    if case["kind"] == "adjoint":  # forward and reverse; carried adjoints and three gradients per facet
        return {"bytes": 2.0 * sweeps * once + F * 14 * R + 24 * F, "flops": 3.5 * case["steps"] * flops}
    return {"bytes": float(sweeps * once + read_out), "flops": float(case["steps"] * flops)}


# --------------------------------------------------------------------------------------------------
# The method in plain torch, FP64 (paper Sec. 2, Sec. 3, App. A; frame-free: tangential quantities
# are global vectors).  It makes the restart states and the reference results.
# --------------------------------------------------------------------------------------------------
def _norm(s):
    """sqrt with derivative 0 at 0."""
    pos = s > 0
    return torch.where(pos, torch.sqrt(torch.where(pos, s, torch.ones_like(s))), torch.zeros_like(s))


class _Reference:
    def __init__(self, spec, mat, bc, par):
        up = lambda a, t=torch.float64: torch.as_tensor(a, device="cuda").to(t)  # noqa: E731
        self.mat, self.N = mat, spec.n_particles
        self.I, self.J, self.tet = (up(a, torch.int64) for a in (spec.facet_pi, spec.facet_pj, spec.tets))
        self.ftet = up(spec.facet_tet, torch.int64)
        x, vtx = up(spec.x), up(spec.facet_vtx).reshape(-1, 3, 3)
        d = x[self.J] - x[self.I]
        self.l = d.norm(dim=1)
        self.n = d / self.l[:, None]
        cen = vtx.mean(1)
        self.cI, self.cJ = cen - x[self.I], cen - x[self.J]
        nc = torch.linalg.cross(vtx[:, 1] - vtx[:, 0], vtx[:, 2] - vtx[:, 0])
        self.A = 0.5 * (self.n * nc).sum(1).abs()
        del vtx, nc, cen
        e = [x[self.tet[:, i]] - x[self.tet[:, 0]] for i in (1, 2, 3)]
        g = [torch.linalg.cross(e[(i + 1) % 3], e[(i + 2) % 3]) for i in range(3)]
        det = (e[0] * g[0]).sum(1)
        self.grad = torch.stack([a / (3.0 * det[:, None]) for a in g], 1)
        m = torch.zeros(self.N, dtype=torch.float64, device="cuda")
        m.index_add_(0, self.tet.reshape(-1), (mat["rho"] / 24.0 * det.abs()).repeat_interleave(4))
        dia = up(spec.diameter)
        self.M = torch.cat([m[:, None].expand(-1, 3), (m * dia * dia / 10.0)[:, None].expand(-1, 3)], 1)
        self.par = [mat[k] for k in ("E0", "alpha", "sigma_t")] if par is None else [up(p) for p in par]
        self.mask, self.vb = up(bc.mask, torch.int64), up(bc.vel)
        # row-sum bound of M^-1 K: translations and rotations of both ends of every facet
        k = mat["E0"] * 1.4 * self.A / self.l
        row = torch.zeros((self.N, 2), dtype=torch.float64, device="cuda")
        for P, c in ((self.I, self.cI), (self.J, self.cJ)):
            c = c.norm(dim=1)
            row.index_add_(0, P, torch.stack([k * (2 + c), k * c * (2 + c)], 1))
        lam = float((row / self.M[:, [0, 3]]).max())
        self.dt = float("%.3g" % (0.9 * 2.0 / math.sqrt(lam)))

    def jump(self, w):
        a, b = w[self.I], w[self.J]
        return b[:, :3] - a[:, :3] + torch.linalg.cross(b[:, 3:], self.cJ) - torch.linalg.cross(a[:, 3:], self.cI)

    def strain(self, w):
        s = self.jump(w) / self.l[:, None]
        sN = (s * self.n).sum(1)
        return sN, s - sN[:, None] * self.n

    def volumetric(self, q):
        u = q[self.tet][:, :, :3]
        return ((u[:, 1:] - u[:, :1]) * self.grad).sum((1, 2))[self.ftet]

    def law(self, eN, eT, dN, dT, eV, tN, tT, emax, par=None):
        """Appendix A, both branches evaluated on safe values and selected by the sign of eN."""
        c, (E0, al, st) = self.mat, par or self.par
        dot = lambda a, b: (a * b).sum(1)  # noqa: E731
        if c["elastic"]:
            return E0 * eN, (al * E0) * eT if np.isscalar(E0) else (al * E0)[:, None] * eT, emax
        col = lambda s: s[:, None]  # noqa: E731
        al_ = al if torch.is_tensor(al) else torch.full_like(eN, al)
        frac = eN > 0
        # A.1 fracture
        one = torch.ones_like(eN)
        fN = torch.where(frac, eN, one)
        aT2 = al_ * dot(eT, eT)
        eff, saT = _norm(fN * fN + aT2), _norm(aT2)
        sn, cs = fN / eff, saT / eff
        s0 = 2.0 * st / (sn + torch.sqrt(sn * sn + 4.0 * al_ / c["r_st"] ** 2 * cs * cs))
        Hs, Ht = c["r_s"] * E0 / al_, 2.0 * E0 * self.l / (c["l_t"] - self.l)
        H0 = Hs + (Ht - Hs) * (torch.atan2(fN, saT) * (2.0 / math.pi)) ** c["n_t"]
        em = torch.maximum(emax, eff)
        sbt = s0 * torch.exp(-H0 * (em - s0 / E0).clamp(min=0.0) / s0)
        pN, pT = eN - dN, eT - dT
        old = _norm(pN * pN + al_ * dot(pT, pT))
        de = (dN * (eN + pN) + al_ * dot(dT, eT + pT)) / (torch.where(frac, eff, one) + old)
        told = _norm(tN * tN + dot(tT, tT) / al_)
        if c["k_t"] > 0:
            raise NotImplementedError("the reload rule is not among the cases")
        t = torch.minimum((told + E0 * de).clamp(min=0.0), sbt)
        r = t / eff
        # A.2 compression, A.3 friction
        kN = torch.where(-tN <= c["sigma_c0"], E0 * one, c["Ed_E0"] * E0 * one)
        cN = tN + kN * dN
        ec0 = c["sigma_c0"] / E0 * one
        ec1, eV0 = c["kc0"] * ec0, c["kc3"] * ec0
        eD = eN - eV
        dv = eV + c["beta"] * eD
        neg = eV <= 0
        rDV = torch.where(neg, -eD.abs() / torch.where(neg, eV - eV0, one), eD.abs() / eV0)
        Hc = (c["Hc0_E0"] - c["Hc1_E0"]) * E0 / (1.0 + c["kc2"] * (rDV - c["kc1"]).clamp(min=0.0)) + c["Hc1_E0"] * E0
        mid = c["sigma_c0"] + (-dv - ec0).clamp(min=0.0) * Hc
        sc1 = c["sigma_c0"] + (ec1 - ec0) * Hc
        late = -dv > ec1
        sbc = torch.where(late, sc1 * torch.exp(torch.where(late, -dv - ec1, 0 * one) * Hc / sc1), mid)
        sbc = torch.where(-dv <= 0, c["sigma_c0"] * one, sbc)
        cN = torch.maximum(cN, -sbc).clamp(max=0.0)
        cT = tT + col(al_ * E0) * dT
        mu = (c["mu0"] - c["mu_inf"]) * c["sigma_N0"]
        sbs = c["r_st"] * st + mu - c["mu_inf"] * cN - mu * torch.exp(cN / c["sigma_N0"])
        tau = _norm(dot(cT, cT))
        slip = tau > sbs
        cT = cT * col(torch.where(slip, sbs / torch.where(slip, tau, one), one))
        return (torch.where(frac, r * eN, cN), torch.where(col(frac), col(al_ * r) * eT, cT),
                torch.where(frac, em, emax))

    def forces(self, tN, tT):
        F = self.A[:, None] * (tN[:, None] * self.n + tT)
        f = torch.zeros((self.N, 6), dtype=torch.float64, device="cuda")
        f = f.index_add(0, self.I, torch.cat([F, torch.linalg.cross(self.cI, F)], 1))
        return f.index_add(0, self.J, -torch.cat([F, torch.linalg.cross(self.cJ, F)], 1))

    def restart(self, q, v, step, strained):
        """State (q, v) with the history of a proportional loading up to q (zero if not strained)."""
        self.q, self.v, self.step0 = torch.as_tensor(q, device="cuda"), torch.as_tensor(v, device="cuda"), step
        F = len(self.l)
        zero, zero3 = torch.zeros(F, dtype=torch.float64, device="cuda"), torch.zeros((F, 3), dtype=torch.float64, device="cuda")
        self.hist = (zero, zero3, zero)
        if strained:
            eN, eT = self.strain(self.q)
            self.hist = self.law(eN, eT, eN, eT, self.volumetric(self.q), zero, zero3, zero)

    def hist5(self):
        tN, tT, em = self.hist
        return torch.cat([tN[:, None], tT, em[:, None]], 1)

    def march(self, steps, par=None):
        """Central difference from the restart state; yields (q, v, v_half, f_old, f) after each step."""
        q, v, (tN, tT, em), dt = self.q, self.v, self.hist, self.dt
        f = self.forces(tN, tT)
        free = self.mask == 0
        bound = torch.where(self.mask == 2, self.vb, torch.zeros_like(self.vb))
        for _ in range(steps):
            vh = torch.where(free, v + (0.5 * dt) * f / self.M, bound)
            q = q + dt * vh
            eN, eT = self.strain(q)
            dN, dT = self.strain(dt * vh)
            tN, tT, em = self.law(eN, eT, dN, dT, self.volumetric(q), tN, tT, em, par)
            f_old, f = f, self.forces(tN, tT)
            v = torch.where(free, vh + (0.5 * dt) * f / self.M, bound)
            self.hist = (tN, tT, em)
            yield q, v, vh, f_old, f


def _exact_adjoint(ref, steps, seeds):
    one = torch.ones_like(ref.l)
    par = [(p * one).requires_grad_() for p in ref.par]
    weight = torch.as_tensor(seeds, device="cuda") * (ref.mask != 0)
    J = 0.0
    for _, _, _, _, f in ref.march(steps, par):
        J = J - (weight * f).sum() / steps  # constant prescribed velocities: reactions are -f
    return J, torch.autograd.grad(J, par)


def exact(case, seed):
    cost = case["steps"] * case["block"] * case["nx"] * case["ny"] * case["nz"]
    if case["kind"] == "adjoint" and cost > 250000:  # every step's intermediates are kept: memory
        return None
    parts = []
    for k in range(case["batch"]):
        b = _build(case, seed, k)
        if case["kind"] == "adjoint":
            J, grads = _exact_adjoint(b.ref, case["steps"], (b.bc.mask == workloads.PRESCRIBED).astype(np.float64))
            return {"objective": J.item(), "grads": [g.cpu().numpy() for g in grads]}
        energy, reaction, wi, we = [], [], 0.0, 0.0
        for q, v, vh, f_old, f in b.ref.march(case["steps"]):
            if case["kind"] == "log":
                dq, mid = b.ref.dt * vh, 0.5 * (f_old + f)
                wi = wi - (mid * dq).sum()
                we = we - (mid * dq * (b.ref.mask != 0)).sum()
                energy.append(torch.stack([we, wi, 0.5 * (b.ref.M * v * v).sum()]))
                reaction.append(torch.cat([(-f * (b.ref.mask == c)).sum(0) for c in (1, 2)]))
        parts.append({"q": q, "v": v, "hist": b.ref.hist5()})
        if energy:
            parts[0] |= {"energy": torch.stack(energy).cpu().numpy(), "reaction": torch.stack(reaction).cpu().numpy()}
        b.ref = None
    return {k: torch.cat([p[k] for p in parts]) if k in "qvhist" else parts[0][k] for k in parts[0]}
