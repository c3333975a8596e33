"""The work that users of this framework have it do, as measurable cases.

A case is a plain dict; `prepare` builds the fluid and the handle a program keeps, `run` makes
one pass through the public entry points (`paper_1806_10841_gb300.adress.AdResS`), `work` counts
what a pass cannot do without and `exact` evaluates the definition in float64 with plain torch
where that is quick.  Every input comes from the seed alone: lattice fluids with vacancies,
jittered centres, random orientations without close contacts, Maxwell-Boltzmann velocities.

Kinds
  block   the thermodynamic-force iteration of an AdResS production run: MD steps with density
          samples every 10 steps and one update of the thermodynamic force, one call
          (`run`); with `all_at` the all-atomistic sampling run of force matching (`step`).
  batch   the same block for many independent replicas in one handle.
  forces  forces, energies and virial of a configuration (lists built on the way): what a
          program asks for on new positions, and the local force engine of the slab
          decomposition.
  rdf     structure and temperature of a snapshot: pair-distance histogram, kinetic energy.
  train   one epoch of the learned coarse-grained force and its held-out predictions.
  fit     the force-matched table from held samples.

A block returns the state as a frame.  On the FP32 mixed path the frame is in single precision,
as trajectory formats store it (its forces are single precision; the double accumulators of
x and v only keep their sums exact); on the FP64 path it is the double state itself.
"""
from __future__ import annotations

import copy
import math

import numpy as np
import torch

from paper_1806_10841_gb300 import adress, inputs

MD_SAMPLE, TF_ALPHA = 10, 0.5
RDF_BINS, RDF_DR = 250, 0.02
FIT_DR, FIT_NMIN = 0.01, 20


# ---------------------------------------------------------------------------- the cases

def _block(M, **kw):
    c = dict(kind="block", fluid="tetra", M=M, precision="fp32", steps=100, scheme=0, respa=1, centers=0,
             net=False, all_at=False)
    c.update(kw)
    return c


def listed():
    return [
        # 1000 molecules: parameter scans and teaching-size systems; a step is a few microseconds
        # of work, so launches and latency count
        dict(_block(1000), name="tetra_4k"),
        # the headline workload: 800k atoms, FP32 mixed
        dict(_block(200_000), name="tetra_800k"),
        # the double-precision path: all-atomistic sampling run for force matching, odd size
        dict(_block(20_011, precision="fp64", all_at=True), name="allatom_80k_fp64"),
        # the double-precision path with the hybrid scheme on the headline fluid
        dict(_block(200_000, precision="fp64", steps=20), name="tetra_800k_fp64"),
        # the water-like fluid (Lennard-Jones + reaction field, long lists)
        dict(_block(64_000, fluid="water", steps=20), name="water_192k"),
        # learned coarse-grained force in every step
        dict(_block(200_000, net=True, steps=50), name="learned_800k"),
        # energy interpolation with multiple time stepping, ragged size
        dict(_block(33_333, scheme=1, respa=2), name="energy_133k"),
        # self-adjusting geometry: 16 moving spheres
        dict(_block(200_000, centers=16), name="spheres_800k"),
        # 64 independent replicas of 500..20000 molecules in one handle
        dict(kind="batch", n=64, m_lo=500, m_hi=20_000, precision="fp32", steps=50, name="replicas_64"),
        # new positions: lists, forces, energies, virial
        dict(kind="forces", fluid="tetra", M=200_000, precision="fp32", scheme=0, name="forces_800k"),
        # structure of a snapshot of the headline fluid
        dict(kind="rdf", M=200_000, precision="fp32", name="rdf_200k"),
        # learned force: one training epoch, then predictions for held-out pairs
        dict(kind="train", samples=300_007, held=30_001, batch=4096, name="train_300k"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    k = rng.choice(["block", "block", "block", "fp64", "water", "net", "centers", "batch", "forces", "forces", "rdf",
                    "train", "fit"])
    if k == "block":
        return _block(_log(rng, 500, 200_000), scheme=rng.choice([0, 0, 1]), respa=rng.choice([1, 1, 2, 4]))
    if k == "fp64":
        return _block(_log(rng, 500, 50_000), precision="fp64", steps=20, all_at=rng.choice([False, True]))
    if k == "water":
        return _block(_log(rng, 1500, 64_000), fluid="water", steps=20)
    if k == "net":
        return _block(_log(rng, 2000, 200_000), net=True, steps=50, respa=rng.choice([1, 1, 4]))
    if k == "centers":
        return _block(_log(rng, 5000, 200_000), centers=rng.choice([1, 3, 16]))
    if k == "batch":
        n = rng.randint(3, 64)
        lo = _log(rng, 500, 3000)
        return dict(kind="batch", n=n, m_lo=lo, m_hi=lo + rng.randint(1, 15_000), precision="fp32", steps=50)
    if k == "forces":
        fluid = rng.choice(["tetra", "tetra", "water"])
        return dict(kind="forces", fluid=fluid, M=_log(rng, 1500 if fluid == "water" else 500, 30_000 if fluid == "water" else 200_000),
                    precision=rng.choice(["fp32", "fp32", "fp64"]), scheme=rng.choice([0, 0, 1]))
    if k == "rdf":
        return dict(kind="rdf", M=_log(rng, 500, 200_000), precision=rng.choice(["fp32", "fp64"]))
    if k == "train":
        return dict(kind="train", samples=_log(rng, 20_000, 300_000), held=_log(rng, 1000, 30_000),
                    batch=rng.choice([512, 1000, 1024, 4096]))
    return dict(kind="fit", samples=_log(rng, 20_000, 1_000_000))


# --------------------------------------------------------------------------- the inputs

def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _rotations(g, n, dev):
    u1, u2, u3 = torch.rand(3, n, generator=g, device=dev, dtype=torch.float64).unbind(0)
    a, b = torch.sqrt(1 - u1), torch.sqrt(u1)
    x, y = a * torch.sin(2 * math.pi * u2), a * torch.cos(2 * math.pi * u2)
    z, w = b * torch.sin(2 * math.pi * u3), b * torch.cos(2 * math.pi * u3)
    return torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - z * w), 2 * (x * z + y * w),
                        2 * (x * y + z * w), 1 - 2 * (x * x + z * z), 2 * (y * z - x * w),
                        2 * (x * z - y * w), 2 * (y * z + x * w), 1 - 2 * (x * x + y * y)], -1).view(n, 3, 3)


def _fluid(s, seed):
    """Positions and velocities (3, N) float64: molecules on lattice sites (vacancies at random),
    centres jittered, orientations random; of two molecules with an atom pair (or centres) too
    close the later one is drawn again."""
    dev = _device()
    g = torch.Generator(device=dev)
    g.manual_seed(int(seed) * 2654435761 % (1 << 62))
    water = s.na == 3
    body = torch.tensor(inputs.water_sites() if water else inputs.tetra_sites(), device=dev, dtype=torch.float64)
    jitter, contact, com_min = (0.01, 0.17, 0.0) if water else (0.2, 0.97, 1.5)
    L = torch.tensor(s.box, device=dev, dtype=torch.float64)
    a = (float(np.prod(s.box)) / s.M) ** (1 / 3)
    n = [max(1, int(math.floor(b / a + 1e-9))) for b in s.box]
    while n[0] * n[1] * n[2] < s.M:
        k = int(np.argmax([b / m for b, m in zip(s.box, n)]))
        n[k] += 1
    nt = torch.tensor(n, device=dev)
    pick = torch.randperm(n[0] * n[1] * n[2], generator=g, device=dev)[:s.M].sort().values
    site = torch.stack([pick // (n[1] * n[2]), pick // n[2] % n[1], pick % n[2]], -1)
    centre0 = (site + 0.5) * (L / nt)
    occ = torch.full((n[0] * n[1] * n[2],), -1, dtype=torch.int64, device=dev)
    occ[pick] = torch.arange(s.M, device=dev)
    off = torch.tensor([(i, j, k) for i in (-1, 0, 1) for j in (-1, 0, 1) for k in (-1, 0, 1) if (i, j, k) != (0, 0, 0)],
                       device=dev)

    def place(m):
        c = centre0[m] + jitter * (2 * torch.rand(len(m), 3, generator=g, device=dev, dtype=torch.float64) - 1)
        return c, c[:, None] + torch.einsum("mij,kj->mki", _rotations(g, len(m), dev), body)

    every = torch.arange(s.M, device=dev)
    com, pos = place(every)
    active = every
    for _ in range(500):
        bad = torch.zeros(s.M, dtype=torch.bool, device=dev)
        for part in active.split(50_000):
            nb = (site[part][:, None] + off) % nt
            b = occ[(nb[..., 0] * n[1] + nb[..., 1]) * n[2] + nb[..., 2]]
            i, j = torch.nonzero((b >= 0) & (b != part[:, None]), as_tuple=True)
            i, j = part[i], b[i, j]
            d = com[i] - com[j]
            d -= L * torch.round(d / L)
            hit = d.square().sum(-1) < com_min ** 2
            d = pos[i][:, :, None] - pos[j][:, None]
            d -= L * torch.round(d / L)
            hit |= (d.square().sum(-1) < contact ** 2).flatten(1).any(1)
            bad[torch.maximum(i, j)[hit]] = True
        active = torch.nonzero(bad)[:, 0]
        if not len(active):
            break
        com[active], pos[active] = place(active)
    else:
        raise RuntimeError("no placement without close contacts")
    if water:  # thermal bond lengths and angles
        pos = pos + 0.0025 * torch.randn(s.M, s.na, 3, generator=g, device=dev, dtype=torch.float64)
    x = torch.remainder(pos.reshape(-1, 3), L)
    x = torch.where(x >= L, x - L, x)
    m = torch.tensor(np.tile(s.mass, s.M), device=dev)[:, None]
    v = torch.randn(s.M * s.na, 3, generator=g, device=dev, dtype=torch.float64) * torch.sqrt(s.kT / m)
    v -= (m * v).sum(0) / m.sum()
    return x.T.contiguous(), v.T.contiguous()


def _system(case):
    kw = {}
    if case.get("scheme"):
        kw["scheme"] = 1
    if case.get("respa", 1) > 1:
        kw["respa_n"] = case["respa"]
    M = case["M"]
    if case.get("fluid") == "water":
        return inputs.scaled_c3(M, **kw) if M != 64_000 else inputs.c3_water(**kw)
    s = inputs.c1_stable(**kw) if M == 1000 else inputs.c2_800k(**kw) if M == 200_000 else inputs.scaled_c2(M, **kw)
    if case.get("all_at"):
        s.d_at = 1e4  # every molecule atomistic
    if case.get("centers"):
        s.d_at, s.d_hy = 0.1 * s.box[2], 0.05 * s.box[2]
        s.tf = np.zeros(int(math.ceil((s.d_at + s.d_hy) / s.tf_dx)) + 2)
    return s


def _network(seed):
    """A smooth repulsive pair force with a weak dependence on the orientations: random hidden
    features, output weights fitted to a soft-core force."""
    rng = np.random.default_rng(seed + 7)
    n = 4000
    feat = np.concatenate([rng.uniform(0.2, 2.3, (n, 1)), np.sort(rng.uniform(-0.59, 0.59, (n, 4)), 1),
                           np.sort(rng.uniform(-0.59, 0.59, (n, 4)), 1)], 1)
    f = 60.0 * (1 - feat[:, 0] / 2.3) ** 2
    mean, std, scale = feat.mean(0), feat.std(0), float(f.std())
    W1 = rng.normal(0, 1 / 3, (64, 9))
    W1[:, 0] *= 3.0
    W1[:, 1:] *= 0.3
    p = dict(W1=W1, b1=rng.normal(0, 0.5, 64), W2=rng.normal(0, 1 / 8, (64, 64)), b2=rng.normal(0, 0.3, 64))

    def silu(z):
        return z / (1 + np.exp(-z))

    h = silu(silu(((feat - mean) / std) @ p["W1"].T + p["b1"]) @ p["W2"].T + p["b2"])
    A = np.concatenate([h, np.ones((n, 1))], 1)
    w = np.linalg.solve(A.T @ A + 1e-2 * np.eye(65), A.T @ (f / scale))
    p["w3"], p["b3"] = w[:64], float(w[64])
    return p, mean, std, scale


def _samples(n, seed):
    """Pairs of tetrahedra at centre distances below the cutoff: features (n, 9) and the projected
    atomistic force between them, float32, as the collection of pair samples gives them."""
    dev = _device()
    g = torch.Generator(device=dev)
    g.manual_seed(int(seed) * 2654435761 % (1 << 62) + 3)
    body = torch.tensor(inputs.tetra_sites(), device=dev, dtype=torch.float64)
    feats, targets, have = [], [], 0
    while have < n:
        m = max(4096, 2 * (n - have))
        u = torch.rand(m, generator=g, device=dev, dtype=torch.float64)
        d = (1.3 ** 3 + u * (2.3 ** 3 - 1.3 ** 3)) ** (1 / 3)
        A = torch.einsum("mij,kj->mki", _rotations(g, m, dev), body)
        B = torch.einsum("mij,kj->mki", _rotations(g, m, dev), body)
        B = B + torch.stack([torch.zeros_like(d), torch.zeros_like(d), d], -1)[:, None]  # e = +z
        r = A[:, :, None] - B[:, None]
        d2 = r.square().sum(-1)
        ok = (d2.flatten(1).min(1).values > 0.9 ** 2)
        ir2 = 1 / d2
        sr6 = ir2 ** 3
        fr = torch.where(d2 < inputs.WCA_RC ** 2, 24 * (2 * sr6 * sr6 - sr6) * ir2, torch.zeros_like(d2))
        t = -(fr * r[..., 2]).sum((1, 2))
        f = torch.cat([d[:, None], A[..., 2].sort(1).values, (-(B[..., 2] - d[:, None])).sort(1).values], 1)
        feats.append(f[ok])
        targets.append(t[ok])
        have += int(ok.sum())
    return (torch.cat(feats)[:n].float().cpu().numpy(), torch.cat(targets)[:n].float().cpu().numpy())


def _handle(systems, precision, x, v):
    sim = adress.AdResS(systems, precision=precision)
    sim.set_state(x, v)
    return sim


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("block", "forces", "rdf"):
        s = _system(case)
        s.seed = 20180628 + seed % 1_000_003
        rng = np.random.default_rng(seed)
        if case.get("centers"):
            s.centers = rng.uniform(0, 1, (case["centers"], 3)) * np.array(s.box)
        x, v = _fluid(s, seed)
        sim = _handle(s, case["precision"], x, v)
        if case.get("net"):
            sim.mlp_set(*_network(seed))
            sim.set_cg_mode(1)
        if kind == "block":
            sim.compute_forces(energies=False)
            sim.check()
        return dict(case=case, sim=sim, rng=rng, centers=s.centers)
    if kind == "batch":
        systems = inputs.replica_batch(case["n"], m_lo=case["m_lo"], m_hi=case["m_hi"])
        for s in systems:
            s.seed = 20180628 + seed % 1_000_003
        st = [_fluid(s, seed + 1000 * r) for r, s in enumerate(systems)]
        sim = _handle(systems, case["precision"], torch.cat([q[0] for q in st], 1), torch.cat([q[1] for q in st], 1))
        sim.compute_forces(energies=False)
        sim.check()
        return dict(case=case, sim=sim)
    s = inputs.scaled_c2(1000)
    sim = adress.AdResS(s, precision="fp32")
    n = case["samples"]
    feat, t = _samples(n + case.get("held", 0), seed)
    sim.mlp_load_samples(feat[:n], t[:n])
    if kind == "train":
        rng = np.random.default_rng(seed)
        sim.mlp_set(dict(W1=rng.normal(0, 1 / 3, (64, 9)), b1=np.zeros(64), W2=rng.normal(0, 1 / 8, (64, 64)),
                         b2=np.zeros(64), w3=rng.normal(0, 1 / 8, 64), b3=float(t[:n].mean() / t[:n].std())),
                    feat[:n].mean(0), feat[:n].std(0) + 1e-3, float(t[:n].std()))
    return dict(case=case, sim=sim, held=feat[n:])


def _frame(sim):
    if sim.precision == "fp64":
        return dict(x=sim.x, v=sim.v, f=sim.f)
    return dict(x=sim.x.float(), v=sim.v.float(), f=sim.f)


def run(state):
    case, sim = state["case"], state["sim"]
    kind = case["kind"]
    if kind in ("block", "batch"):
        if case.get("all_at"):
            sim.step(case["steps"])
            return _frame(sim)
        if case.get("centers"):  # the region follows its centres: a tenth of a sigma per block
            state["centers"] = state["centers"] + state["rng"].normal(0, 0.1 / math.sqrt(3.0), state["centers"].shape)
            sim.set_centers(state["centers"])
        sim.run(case["steps"], sample_every=MD_SAMPLE, tf_update=True, alpha=TF_ALPHA)
        return dict(_frame(sim), tf=sim.get_tf())
    if kind == "forces":
        e = sim.compute_forces(energies=True)
        return dict(f=sim.f, e=e)
    if kind == "rdf":
        counts = sim.rdf_counts(RDF_BINS, RDF_DR)
        ke, p = sim.kinetic()
        return dict(counts=counts, ke=ke, p=p)
    if kind == "train":
        loss = sim.mlp_train(epochs=1, batch=case["batch"], lr=2e-3)
        held = state["held"]
        swapped = held[:, [0, 5, 6, 7, 8, 1, 2, 3, 4]]
        y = 0.5 * (sim.mlp_forward(held) + sim.mlp_forward(swapped))
        return dict(loss=loss, params=sim.mlp_flatten(sim.mlp_get()), y=y.astype(np.float32))
    F, V = sim.cg_fit(FIT_DR, FIT_NMIN)
    return dict(F=F, V=V)


# ------------------------------------------------------------------------------ the work

def _force_flops(s, spheres=0):
    """Pair interactions inside the cutoffs at the fluid's mean density, each pair once."""
    rho = s.M / float(np.prod(s.box))
    if spheres:
        hr = min(1.0, spheres * 4 / 3 * math.pi * (s.d_at + s.d_hy) ** 3 / float(np.prod(s.box)))
    else:
        hr = min(1.0, 2 * (s.d_at + s.d_hy) / s.box[0])
    at = hr * s.N / 2 * (rho * s.na) * 4 / 3 * math.pi * s.rc_at ** 3
    cg = (1 - 0.66 * hr) * s.M / 2 * rho * 4 / 3 * math.pi * s.rc_cg ** 3
    if s.d_at > s.box[0]:
        cg = 0.0
    return 35 * at + 55 * cg + 40 * s.M * len(s.bonds)


def work(case):
    kind = case["kind"]
    if kind in ("block", "forces", "rdf"):
        s = _system(case)
        fb = 8 if case["precision"] == "fp64" else 4
        if kind == "block":  # every step reads and writes x and v of every atom
            flops = _force_flops(s, case["centers"]) + 60 * s.N + (2 * 2 * (9 * 64 + 64 * 64 + 64) * 2.3 * s.M if case["net"] else 0)
            return dict(bytes=96.0 * s.N * case["steps"], flops=flops * case["steps"])
        if kind == "forces":
            return dict(bytes=(24.0 + 3 * fb) * s.N, flops=_force_flops(s))
        rho = s.M / float(np.prod(s.box))
        return dict(bytes=48.0 * s.N + 8.0 * RDF_BINS, flops=10.0 * s.M / 2 * rho * 4 / 3 * math.pi * (RDF_BINS * RDF_DR) ** 3)
    if kind == "batch":
        m = (case["m_hi"] - case["m_lo"]) / math.log(case["m_hi"] / case["m_lo"]) * case["n"]  # mean of log-uniform sizes
        return dict(bytes=96.0 * 4 * m * case["steps"], flops=4 * m * 150.0 * case["steps"])
    if kind == "train":
        per = 2.0 * (9 * 64 + 64 * 64 + 64)
        return dict(bytes=40.0 * case["samples"] + 40.0 * case["held"], flops=3 * per * case["samples"] + 2 * per * case["held"])
    return dict(bytes=8.0 * case["samples"] + 16.0 * 2301, flops=4.0 * case["samples"])


# ------------------------------------------------- the definition in float64, plain torch

def _minimg(d, L):
    return d - L * torch.round(d / L)


def _mapping(s, x, L):
    """Centres of mass, offsets and resolution of atoms x (N, 3)."""
    m = torch.tensor(s.mass, device=x.device)
    xm = x.view(s.M, s.na, 3)
    d0 = _minimg(xm - xm[:, :1], L)
    c = (m[:, None] * d0).sum(1) / m.sum()
    R = torch.remainder(xm[:, 0] + c, L)
    dx = _minimg(R[:, 0] - s.xc, L[0])
    d = dx.abs()
    lam = torch.where(d < s.d_at, 1.0, torch.where(d >= s.d_at + s.d_hy, 0.0, torch.cos(0.5 * math.pi * (d - s.d_at) / s.d_hy) ** 2))
    return R, d0 - c[:, None], dx, lam


def _pairs(R, L, cut):
    """All pairs a < b of centres within cut."""
    Rf, Lf = R.float(), L.float()
    out = []
    step = max(1, 200_000_000 // len(R))
    for a0 in range(0, len(R), step):
        r2 = torch.zeros(min(step, len(R) - a0), len(R) - a0, device=R.device)
        for d in range(3):
            t = (Rf[a0:a0 + step, d, None] - Rf[None, a0:, d]).abs_()
            t = torch.minimum(t, Lf[d] - t)
            r2.addcmul_(t, t)
        a, b = torch.nonzero(r2 < (cut + 1e-3) ** 2, as_tuple=True)
        keep = b > a
        out.append(torch.stack([a[keep] + a0, b[keep] + a0]))
    return torch.cat(out, 1)


def _exact_forces(s, x, pairs, sw=1.0):
    """Conservative forces of Eq. 1 at positions x (N, 3), with the slow forces at weight sw;
    energies (E_at, E_cg, E_bond, virial)."""
    dev = x.device
    L = torch.tensor(s.box, device=dev, dtype=torch.float64)
    R, o, dx, lam = _mapping(s, x, L)
    frac = torch.tensor(s.mass / s.mass.sum(), device=dev)
    f = torch.zeros_like(x).view(s.M, s.na, 3)
    a, b = pairs
    dR = _minimg(R[a] - R[b], L)
    w = lam[a] * lam[b]
    r2 = dR.square().sum(-1)
    # atomistic part
    p = torch.nonzero((w > 0) & (r2 < (s.rc_at + 2 * s.r_ext + 0.5) ** 2))[:, 0]
    pa, pb = a[p], b[p]
    d = dR[p][:, None, None] + o[pa][:, :, None] - o[pb][:, None]
    d2 = d.square().sum(-1)
    if s.nb_model:
        eps = torch.tensor(np.sqrt(np.outer(s.lj_eps, s.lj_eps)), device=dev)
        sg6 = torch.tensor((0.5 * np.add.outer(s.lj_sig, s.lj_sig)) ** 6, device=dev)
        qq = torch.tensor(s.coulomb_f * np.outer(s.charge, s.charge), device=dev)
        krf = (s.eps_rf - 1) / ((2 * s.eps_rf + 1) * s.rc_at ** 3)
        crf = 1 / s.rc_at + krf * s.rc_at ** 2
        ir2 = 1 / d2
        t6 = sg6 * ir2 ** 3
        tc = sg6 / s.rc_at ** 6
        fr = 24 * eps * (2 * t6 * t6 - t6) * ir2 + qq * (ir2.sqrt() * ir2 - 2 * krf)
        e = 4 * eps * (t6 * t6 - t6 - tc * tc + tc) + qq * (ir2.sqrt() + krf * d2 - crf)
    else:
        ir2 = 1 / d2
        t6 = s.sigma ** 6 * ir2 ** 3
        fr = 24 * s.eps * (2 * t6 * t6 - t6) * ir2
        e = 4 * s.eps * (t6 * t6 - t6) + s.eps
    mask = torch.where(d2 < s.rc_at ** 2, w[p][:, None, None], torch.zeros_like(d2))
    fr = fr * mask
    F = fr[..., None] * d
    f.index_add_(0, pa, F.sum(2))
    f.index_add_(0, pb, -F.sum(1))
    e_at, vir = (e * mask).sum(), (fr * d2).sum()
    # coarse-grained part
    q = torch.nonzero((w < 1) & (r2 < s.rc_cg ** 2))[:, 0]
    r = r2[q].sqrt()
    u = r / s.cg_dr
    k = u.long().clamp(max=s.cg_n - 1)
    t = u - k
    tF, tV = torch.tensor(s.cg_F, device=dev), torch.tensor(s.cg_V, device=dev)
    W = 1 - w[q]
    Fc = W * (tF[k] * (1 - t) + tF[k + 1] * t)
    e_cg = (W * (tV[k] * (1 - t) + tV[k + 1] * t)).sum()
    vir = vir + (Fc * r).sum()
    G = (sw * Fc / r)[:, None, None] * dR[q][:, None] * frac[:, None]
    f.index_add_(0, a[q], G)
    f.index_add_(0, b[q], -G)
    # bonded terms
    e_b = torch.zeros((), device=dev, dtype=torch.float64)
    for i, j in np.asarray(s.bonds).reshape(-1, 2).tolist():
        bd = o[:, i] - o[:, j]
        b2 = bd.square().sum(-1)
        if s.bond_model == 1:
            l = b2.sqrt()
            bf = -s.bond_k * (l - s.bond_r0) / l
            e_b = e_b + (0.5 * s.bond_k * (l - s.bond_r0) ** 2).sum()
        else:
            bf = -s.fene_k / (1 - b2 / s.fene_r0 ** 2)
            e_b = e_b - (0.5 * s.fene_k * s.fene_r0 ** 2 * torch.log(1 - b2 / s.fene_r0 ** 2)).sum()
            if s.intra_wca:
                t6 = (s.sigma ** 2 / b2) ** 3
                inside = b2 < s.rc_at ** 2
                bf = bf + torch.where(inside, 24 * s.eps * (2 * t6 * t6 - t6) / b2, torch.zeros_like(b2))
                e_b = e_b + torch.where(inside, 4 * s.eps * (t6 * t6 - t6) + s.eps, torch.zeros_like(b2)).sum()
        f[:, i] += bf[:, None] * bd
        f[:, j] -= bf[:, None] * bd
        vir = vir + (bf * b2).sum()
    if s.bond_model == 1 and s.angles is not None:
        for i, j, k in np.asarray(s.angles).reshape(-1, 3).tolist():
            with torch.enable_grad():
                uu = (o[:, i] - o[:, j]).requires_grad_(True)
                vv = (o[:, k] - o[:, j]).requires_grad_(True)
                th = torch.acos((uu * vv).sum(-1) / (uu.norm(dim=-1) * vv.norm(dim=-1)))
                E = (0.5 * s.angle_k * (th - s.angle_theta0) ** 2).sum()
                gu, gv = torch.autograd.grad(E, (uu, vv))
            f[:, i] -= gu
            f[:, k] -= gv
            f[:, j] += gu + gv
            e_b = e_b + E.detach()
            vir = vir - (uu.detach() * gu + vv.detach() * gv).sum()
    # thermodynamic force
    if len(s.tf):
        ad = dx.abs()
        u = ad / s.tf_dx
        k = u.long()
        tf = torch.tensor(np.concatenate([s.tf, [0.0, 0.0]]), device=dev)
        kc = k.clamp(max=len(s.tf))
        T = torch.where(k + 1 < len(s.tf), tf[kc] * (1 - (u - k)) + tf[kc + 1] * (u - k), torch.zeros_like(u))
        T = torch.where((ad >= s.d_at) & (ad < s.d_at + s.d_hy), T, torch.zeros_like(T)) * sw
        f[:, :, 0] += frac * (torch.where(dx < 0, -T, T))[:, None]
    return f.view(-1, 3), (e_at, e_cg, e_b, vir)


def _philox(N, step, replica, block, seed, dev):
    """Philox4x32-10 (Salmon et al. 2011): counter (atom, step lo, step hi, 2 replica + block)."""
    M32 = 0xFFFFFFFF
    c = [torch.arange(N, device=dev)] + [torch.full((N,), v, dtype=torch.int64, device=dev)
                                         for v in (step & M32, step >> 32, 2 * replica + block)]
    k0, k1 = seed & M32, seed >> 32

    def mul(m, v):  # high and low words of a 32 x 32 bit product
        lo = m * (v & 0xFFFF)
        hi = m * (v >> 16) + (lo >> 16)
        return (hi >> 16) & M32, ((hi << 16) | (lo & 0xFFFF)) & M32

    for r in range(10):
        h0, l0 = mul(0xD2511F53, c[0])
        h1, l1 = mul(0xCD9E8D57, c[2])
        c = [h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0]
        k0, k1 = (k0 + 0x9E3779B9) & M32, (k1 + 0xBB67AE85) & M32
    return torch.stack(c[:3], -1)


def _noise(s, step, precision, dev):
    c = _philox(s.N, step, 0, 0, s.seed, dev)
    if precision == "fp32":
        return (c >> 8).double() / 16777216.0
    return ((c << 21) | (_philox(s.N, step, 0, 1, s.seed, dev) >> 11)).double() / 9007199254740992.0


def _exact_block(s, case, x, v):
    dev = x.device
    L = torch.tensor(s.box, device=dev, dtype=torch.float64)
    m = torch.tensor(np.tile(s.mass, s.M), device=dev)[:, None]
    amp = torch.sqrt(24 * s.gamma * s.kT * m / s.dt)
    n = max(1, s.respa_n)

    def weight(step):
        return float(n) if n > 1 and step % n == 0 else 0.0 if n > 1 else 1.0

    cut = max(s.rc_cg, s.rc_at + 2 * s.r_ext) + (0.05 if s.nb_model else 1.0)
    hist, samples = torch.zeros(len(s.tf), dtype=torch.float64, device=dev), 0
    pairs = _pairs(_mapping(s, x, L)[0], L, cut)
    f, _ = _exact_forces(s, x, pairs, weight(0))
    for k in range(case["steps"]):
        v = v + 0.5 * s.dt / m * f
        x = x + s.dt * v
        x = torch.where(x < 0, x + L, x)
        x = torch.where(x >= L, x - L, x)
        if k % 10 == 9:
            R, _, dx, _ = _mapping(s, x, L)
            pairs = _pairs(R, L, cut)
            if not case["all_at"] and (k + 1) % MD_SAMPLE == 0:
                b = torch.floor(dx.abs() / s.tf_dx).long()
                hist += torch.bincount(b[b < len(s.tf)], minlength=len(s.tf)).double()
                samples += 1
        f, _ = _exact_forces(s, x, pairs, weight(k + 1))
        f = f - s.gamma * m * v + amp * (_noise(s, k + 1, case["precision"], dev) - 0.5)
        v = v + 0.5 * s.dt / m * f
    out = dict(x=x.T, v=v.T, f=f.T)
    if not case["all_at"]:
        rho = hist.cpu().numpy() / (samples * 2 * s.tf_dx * s.box[1] * s.box[2])
        g = np.concatenate([[0.0], np.diff(rho) / s.tf_dx])
        tf = np.array(s.tf, dtype=np.float64)
        for k in range(len(tf)):
            if s.d_at <= k * s.tf_dx <= s.d_at + s.d_hy:
                tf[k] -= TF_ALPHA * g[max(0, k - 1):k + 2].mean()
        out["tf"] = tf
    return out


def _exact_fit(feat, target, s):
    d, t = feat[:, 0].astype(np.float64), target.astype(np.float64)
    nb = int(math.ceil(s.rc_cg / FIT_DR))
    j = np.floor(d / FIT_DR).astype(np.int64)
    keep = j < nb
    num, cnt = np.bincount(j[keep], t[keep], nb), np.bincount(j[keep], minlength=nb)
    pop = np.nonzero(cnt >= FIT_NMIN)[0]
    mean, centre = num[pop] / cnt[pop], (pop + 0.5) * FIT_DR
    r = np.arange(len(s.cg_F)) * s.cg_dr
    F = np.where(r < s.rc_cg, np.interp(r, centre, mean) - np.interp(s.rc_cg, centre, mean), 0.0)
    V = np.concatenate([np.cumsum((0.5 * (F[:-1] + F[1:]) * s.cg_dr)[::-1])[::-1], [0.0]])
    return dict(F=F, V=V)


def exact(case, seed):
    kind = case["kind"]
    if kind == "fit":
        feat, t = _samples(case["samples"], seed)
        return _exact_fit(feat, t, inputs.scaled_c2(1000))
    if kind == "rdf":
        s = _system(case)
        _, v = _fluid(s, seed)
        m = torch.tensor(np.tile(s.mass, s.M), device=v.device)
        return dict(counts=None, ke=float((0.5 * m * v.square().sum(0)).sum()), p=None)
    if kind not in ("block", "forces") or case.get("scheme") or case.get("net") or case.get("centers"):
        return None  # other models: their whole trajectories, without a short definition here
    if kind == "block" and case["M"] * case["steps"] > 2_500_000:
        return None  # over twenty seconds of dense pair searches
    s = copy.copy(_system(case))
    s.seed = 20180628 + seed % 1_000_003
    x, v = _fluid(s, seed)
    x, v = x.T.contiguous(), v.T.contiguous()
    with torch.no_grad():
        if kind == "block":
            return _exact_block(s, case, x, v)
        L = torch.tensor(s.box, device=x.device, dtype=torch.float64)
        cut = max(s.rc_cg, s.rc_at + 2 * s.r_ext)
        f, e = _exact_forces(s, x, _pairs(_mapping(s, x, L)[0], L, cut), float(max(1, s.respa_n)))
    return dict(f=f.T, e={k: float(w) for k, w in zip(("E_at", "E_cg", "E_bond", "virial"), e)})
