"""Measured cases of the library: the calls a simulation makes, over the range of its workloads.

Kinds of case (field "kind"):
  transform   rfft3d then irfft3d of real fields: the stand-alone spectral primitive
  residual    stress_residual: spectrum, mean stress and equilibrium residual of a given stress field
  increment   one mechanical increment from a checkpoint held on the device (the state is put back with
              set_fields / set_scalars, as a run with step control does when it repeats an increment), then the
              fields a program reads after it
  drx         what follows an increment: nucleation and the phase-field steps with their statistics, from a
              checkpoint in the DRX regime
  gradient    the calibration's step: stress-strain curve and its gradient with respect to (k1, k2, tau0, n)

Microstructures are periodic Voronoi polycrystals with random orientations, copper constants and the strain
increments of the workloads in paper_1509_04953_gb300/synth.py. exact() restates each path in 64-bit torch.
"""
from __future__ import annotations

import ctypes
import dataclasses
import math

import numpy as np
import torch

from paper_1509_04953_gb300 import autograd, evp, synth


def listed():
    return [
        # the smallest call: a 16^3 parity-size transform, all launch latency
        dict(name="transform_f32_16", kind="transform", n=16, fields=6, dtype="float32"),
        # the spectral primitive at the headline size in the reference precision
        dict(name="transform_f64_128", kind="transform", n=128, fields=6, dtype="float64"),
        # the equilibrium check of a stress field at the headline size
        dict(name="residual_f32_128", kind="residual", n=128, dtype="float32"),
        # a small mixed-precision run (the calibration's grid): many short launches per increment
        dict(name="increment_mixed_32", kind="increment", n=32, grains=27, precision="mixed", scheme="basic",
             law="power", history=4),
        # the headline workload's increment
        dict(name="increment_mixed_128", kind="increment", n=128, grains=256, precision="mixed", scheme="basic",
             law="power", history=5),
        # the large workload's increment
        dict(name="increment_mixed_256", kind="increment", n=256, grains=1024, precision="mixed", scheme="basic",
             law="power", history=2),
        # the FP64 coupled workload's increment
        dict(name="increment_fp64_64", kind="increment", n=64, grains=64, precision="fp64", scheme="basic",
             law="power", history=3),
        # the augmented Lagrangian, the solver the paper names, at the headline size
        dict(name="al_mixed_128", kind="increment", n=128, grains=256, precision="mixed", scheme="al", law="power",
             history=5),
        # the paper's own dislocation law under that solver
        dict(name="al_ma_roters_mixed_64", kind="increment", n=64, grains=64, precision="mixed", scheme="al", law="mr",
             history=3),
        # nucleation and five phase-field steps at the headline size
        dict(name="drx_mixed_128", kind="drx", n=128, grains=256, precision="mixed", refine=1, kmax=8, steps=5),
        # the same on the 2:1 phase-field grid in FP64
        dict(name="drx_fp64_64_refined", kind="drx", n=64, grains=64, precision="fp64", refine=2, kmax=8, steps=5),
        # forward and reverse sweep of the differentiation workload's grid, checkpointed
        dict(name="gradient_fp64_32", kind="gradient", n=32, grains=27, precision="fp64", increments=2,
             checkpoint_every=1),
    ]


def _log_choice(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["transform", "residual", "increment", "increment", "increment", "drx", "drx", "gradient"])
    if kind == "transform":
        return dict(kind=kind, n=rng.choice([16, 32, 64, 128, 256]), fields=rng.randint(1, 6),
                    dtype=rng.choice(["float32", "float64"]))
    if kind == "residual":
        return dict(kind=kind, n=rng.choice([16, 32, 64, 128, 256]), dtype=rng.choice(["float32", "float64"]))
    if kind == "gradient":
        n = rng.choice([16, 32])
        t = 2 if n == 32 else rng.randint(2, 5)
        return dict(kind=kind, n=n, grains=_log_choice(rng, 5, 61), precision="fp64", increments=t,
                    checkpoint_every=rng.randint(1, t))
    if kind == "drx":
        refine = rng.choice([1, 1, 2])
        return dict(kind=kind, n=rng.choice([16, 32, 64] if refine == 2 else [16, 32, 64, 128]),
                    grains=_log_choice(rng, 7, 300), precision=rng.choice(["mixed", "fp64"]), refine=refine,
                    kmax=rng.choice([8, 8, 5, 2]), steps=rng.randint(1, 10))
    precision = rng.choice(["mixed", "mixed", "mixed_fast", "fp64"])
    law = rng.choice(["power", "power", "mr"])
    scheme = "al" if law == "mr" else rng.choice(["basic", "al"])
    n = rng.choice([32, 64] if precision == "fp64" or law == "mr" else [32, 64, 128])
    return dict(kind=kind, n=n, grains=_log_choice(rng, 9, 2 * n), precision=precision, scheme=scheme, law=law,
                history=rng.randint(2, 5))


# ---- inputs, from the seed alone ----

def _material(case):
    return synth.ma_roters_material() if case.get("law") == "mr" else synth.Material()


def _grains(case, seed):
    n, grains = case["n"], case["grains"]
    return synth.voronoi_seeds(n, grains, seed), synth.orientations(grains, seed)


def _loading(case):
    """(dE33, dt) of an increment: the workloads' 1e-3 per second; 6e-4 per 0.6 s on the large grid; the Ma-Roters
    law is run at 1e-3 per 0.625 s."""
    if case.get("law") == "mr":
        return -1.0e-3, 0.625
    return (-6.0e-4, 0.6) if case["n"] >= 256 else (-1.0e-3, 1.0)


def _fields(case, seed):
    """Random fields as a stress field has them: a mean and fluctuations of the same order."""
    n, f = case["n"], case.get("fields", 6)
    gen = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.randn((f, n, n, n), generator=gen, device="cuda", dtype=torch.float64) * 50.0
    x += torch.randn((f, 1, 1, 1), generator=gen, device="cuda", dtype=torch.float64) * 30.0
    return x.to(getattr(torch, case["dtype"]))


def _drx_inputs(case, seed, mat):
    """Density per slip system (a tenth to a half of the critical level over twelve) and nucleation strengths
    (Weibull), per voxel."""
    n3 = case["n"] ** 3
    gen = torch.Generator(device="cuda").manual_seed(seed)
    rho = (0.1 + 0.35 * torch.rand(n3, generator=gen, device="cuda", dtype=torch.float64)) * mat.kc / 12.0
    u = torch.rand(n3, generator=gen, device="cuda", dtype=torch.float64)
    kappa = mat.kc * (-torch.log1p(-u)) ** (1.0 / mat.q)
    t = torch.float64 if case["precision"] == "fp64" else torch.float32
    return rho.to(t).expand(12, n3).contiguous(), kappa


def _theta(case, seed):
    mat = synth.Material()
    rng = np.random.default_rng(seed)
    return torch.tensor([getattr(mat, p) * (1.0 + 0.05 * rng.uniform(-1, 1)) for p in autograd.PARAMS],
                        dtype=torch.float64)


WARM_STEPS = 20   # phase-field steps before the checkpoint of a drx case: diffuse boundaries from the sharp start


class _Checkpoint:
    """The named fields and the scalars of a solver, in one device buffer, to be put back before each pass."""

    def __init__(self, s, names):
        self.s = s
        self.mask = 0
        for name in names:
            self.mask |= evp.FIELDS[name]
        nb = ctypes.c_size_t(0)
        s._check("evp_fields_bytes", evp.load().evp_fields_bytes(s.h, self.mask, ctypes.byref(nb)))
        self.buf = torch.empty(nb.value, dtype=torch.uint8, device="cuda")
        s._check("get_fields", evp.load().get_fields(s.h, self.mask, self.buf.data_ptr(), nb.value, 1))
        self.scalars = s.scalars()
        self.leff = s.leff

    def restore(self):
        s = self.s
        s._check("set_fields", evp.load().set_fields(s.h, self.mask, self.buf.data_ptr(), self.buf.numel(), 1))
        s.set_scalars(**self.scalars)
        s.leff = self.leff


def _set_device(s, name, t):
    s._check("set_fields", evp.load().set_fields(s.h, evp.FIELDS[name], t.data_ptr(), t.numel() * t.element_size(), 1))


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("transform", "residual"):
        return dict(case=case, x=_fields(case, seed))
    seeds, quat = _grains(case, seed)
    n, grains, mat = case["n"], case["grains"], _material(case)
    g0 = evp.voronoi(n, seeds).cpu().numpy()
    dE33, dt = _loading(case)
    if kind == "gradient":
        setup = autograd.CurveSetup(n=n, grains=grains, grain_id=g0, quat=quat, material=mat, seed=seed,
                                    increments=case["increments"], dE33=dE33, dt=dt, precision=case["precision"],
                                    checkpoint_every=case["checkpoint_every"])
        target = torch.tensor([-50.0 - 4.0 * i for i in range(case["increments"])], dtype=torch.float64)
        return dict(case=case, setup=setup, theta=_theta(case, seed).requires_grad_(True), target=target)
    if kind == "drx":
        s = evp.Solver(n, grains, g0, quat, mat, seed, precision=case["precision"], kmax=case["kmax"],
                       pf_refine=case["refine"])
        rho, kappa = _drx_inputs(case, seed, mat)
        _set_device(s, "rho", rho)
        _set_device(s, "kappa", kappa)
        s.pf_step(WARM_STEPS)
        return dict(case=case, s=s, ck=_Checkpoint(s, ("rho", "kappa", "g", "draws", "ids", "eta")))
    mr = case["law"] == "mr"
    tol = 1e-8 if case["precision"] == "fp64" else 5e-6 if mr else 1e-6
    s = evp.Solver(n, grains, g0, quat, mat, seed, precision=case["precision"], scheme=case["scheme"], law=case["law"],
                   al_scale=8.0 if mr else 6.0, tol=tol, max_iter=5000)
    for _ in range(case["history"]):
        s.increment(dE33, dt)
    names = ("sig", "epsp", "epse", "deps", "rho") + (("gnd3",) if mr else ())
    return dict(case=case, s=s, ck=_Checkpoint(s, names), load=(dE33, dt))


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "transform":
        return {"back": evp.irfft3d(evp.rfft3d(state["x"]))}
    if kind == "residual":
        spec, out = evp.stress_residual(state["x"])
        return {"spec": spec, "out": out}
    if kind == "gradient":
        curve = autograd.stress_strain_curve(state["theta"], state["setup"])
        loss = ((curve - state["target"]) ** 2).sum()
        grad, = torch.autograd.grad(loss, state["theta"])
        return {"curve": curve.detach(), "grad": grad}
    s = state["s"]
    state["ck"].restore()
    if kind == "drx":
        _, nuclei = s.nucleate(0)
        _, ps = s.pf_step(case["steps"])
        out = {f: s.get_device(f) for f in ("ids", "eta", "g", "rho", "k")}
        out.update(nuclei=nuclei, F_tot=ps.F_tot, X_rex=ps.X_rex, n_grains=ps.n_grains, overflow=ps.overflow)
        return out
    _, st = s.increment(*state["load"])
    out = {f: s.get_device(f) for f in ("sig", "epsp", "epse", "rho") + (("gnd3",) if case["law"] == "mr" else ())}
    out.update(sig_mean=np.array(st.sig_mean, dtype=s.dtype), E=np.array(st.E, dtype=s.dtype))
    return out


ITERATIONS = 100   # fixed-point iterations counted in work() for one increment (25 with the augmented Lagrangian)


def work(case):
    """Inputs read once, outputs written once; the arithmetic of the transforms and of one residual evaluation per
    voxel and iteration (an increment's iteration count depends on its input: a nominal one is counted)."""
    kind, n = case["kind"], case["n"]
    n3, h = n ** 3, n * n * (n // 2 + 1)
    fft = 2.5 * n3 * math.log2(n3)   # one real transform
    if kind in ("transform", "residual"):
        t = 8 if case["dtype"] == "float64" else 4
        f = case.get("fields", 6)
        if kind == "transform":
            return dict(bytes=2.0 * f * n3 * t, flops=2 * f * fft)
        return dict(bytes=6.0 * (n3 + 2 * h) * t + 56, flops=6 * fft + 40.0 * h)
    t = 8 if case["precision"] == "fp64" else 4
    if kind == "drx":
        m3 = (case["refine"] * n) ** 3
        per = 2.0 * (4 + t)   # about two order parameters per point: read once, written once
        return dict(bytes=2 * per * m3 + n3 * (12.0 * t + 24), flops=60.0 * 3 * case["steps"] * m3)
    iteration = 12 * fft + n3 * (540.0 + 150.0)
    if kind == "gradient":
        return dict(bytes=n3 * 4.0 + 12 * n3 * t, flops=3 * case["increments"] * ITERATIONS * iteration)
    state = 36 + (36 if case["law"] == "mr" else 0)
    its = 25 if case["scheme"] == "al" else ITERATIONS
    return dict(bytes=2.0 * state * n3 * t + 4 * n3, flops=its * iteration)


# ---- the same results in 64-bit torch ----

def _voronoi64(n, seeds):
    s = torch.as_tensor(seeds, device="cuda")
    c = (torch.arange(n, device="cuda") << 16) + 32768
    best = torch.full((n, n, n), 2 ** 62, dtype=torch.int64, device="cuda")
    ids = torch.zeros((n, n, n), dtype=torch.int64, device="cuda")
    for g in range(s.shape[0]):
        d = (c[None] - s[g][:, None]).abs() % (n << 16)
        d = torch.minimum(d, (n << 16) - d) ** 2
        dd = d[2][:, None, None] + d[1][None, :, None] + d[0][None, None, :]
        ids = torch.where(dd < best, g, ids)
        best = torch.minimum(best, dd)
    return ids.reshape(-1)


_PAIRS = [(0, 0), (1, 1), (2, 2), (1, 2), (0, 2), (0, 1)]   # Mandel order, sqrt2 on the shears


def _mandel(t):
    return torch.stack([t[..., i, j] * (1.0 if i == j else math.sqrt(2.0)) for i, j in _PAIRS], -1)


def _tables64(mat, quat):
    """Per grain: compliance (6 x 6) and Schmid vectors (12 x 6) in the sample frame."""
    q = torch.tensor(quat, dtype=torch.float64)
    q = q / q.norm(dim=1, keepdim=True)
    w, x, y, z = q.T
    R = torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
                     2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
                     2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)], 1).reshape(-1, 3, 3)
    Q = torch.empty(R.shape[0], 6, 6, dtype=torch.float64)
    for c, (i, j) in enumerate(_PAIRS):
        B = torch.zeros(3, 3, dtype=torch.float64)
        B[i, j] = B[j, i] = 1.0 if i == j else 1.0 / math.sqrt(2.0)
        Q[:, :, c] = _mandel(R @ B @ R.transpose(1, 2))
    C = torch.diag(torch.tensor([mat.C11 - mat.C12] * 3 + [2 * mat.C44] * 3, dtype=torch.float64))
    C[:3, :3] += mat.C12
    schmid = []
    for nx, ny, nz in [(1, 1, 1), (-1, 1, 1), (1, -1, 1), (1, 1, -1)]:
        for d in [(0, 1, -1), (0, 1, 1), (1, 0, -1), (1, 0, 1), (1, -1, 0), (1, 1, 0)]:
            if nx * d[0] + ny * d[1] + nz * d[2] == 0:
                a = torch.tensor([nx, ny, nz], dtype=torch.float64) / math.sqrt(3.0)
                b = torch.tensor(d, dtype=torch.float64) / math.sqrt(2.0)
                schmid.append(_mandel(0.5 * (torch.outer(a, b) + torch.outer(b, a))))
    m = torch.stack(schmid)
    return (Q @ torch.linalg.inv(C) @ Q.transpose(1, 2)).cuda(), (m @ Q.transpose(1, 2)).cuda()


class _Mechanics64:
    """Power-law increments in FP64, solved by the augmented Lagrangian to round-off (the solution does not depend
    on the scheme)."""

    def __init__(self, case, seed, mat):
        seeds, quat = _grains(case, seed)
        self.n, self.mat = case["n"], mat
        v = self.n ** 3
        g = _voronoi64(self.n, seeds)
        S, M = _tables64(mat, quat)
        self.S, self.M = S[g], M[g]
        z = lambda c: torch.zeros((v, c), dtype=torch.float64, device="cuda")  # noqa: E731
        self.sig, self.ee, self.ep, self.de = z(6), z(6), z(6), z(6)
        self.rho = z(12) + mat.rho0
        self.E, self.dE = np.zeros(6), None
        self.mu0 = mat.mu / 6.0
        self.lam0 = mat.lam + 2.0 * mat.mu / 3.0 - 2.0 * self.mu0 / 3.0
        C0 = 2 * self.mu0 * torch.eye(6, dtype=torch.float64, device="cuda")
        C0[:3, :3] += self.lam0
        self.C0, self.S0 = C0, torch.linalg.inv(C0)
        k = torch.fft.fftfreq(self.n, 1.0 / self.n, dtype=torch.float64, device="cuda")
        kx = torch.arange(self.n // 2 + 1, dtype=torch.float64, device="cuda")
        xi = torch.stack(torch.broadcast_tensors(kx[None, None, :], k[None, :, None], k[:, None, None]), -1)
        half = self.n // 2
        self.nyq = (xi.abs() == half).any(-1)
        nn = xi.pow(2).sum(-1, keepdim=True).sqrt()
        self.dir = xi / torch.where(nn == 0, 1.0, nn)

    def _rates(self, M, sig, tauc, dt):
        m = self.mat
        x = torch.einsum("vai,vi->va", M, sig) / tauc[:, None]
        p = x.abs() ** (m.n - 1)
        gd = m.gdot0 * p * x
        slope = m.n * m.gdot0 * p / tauc[:, None]
        pot = dt * m.gdot0 * tauc / (m.n + 1) * (p * x * x).sum(1)
        return gd, slope, pot

    def _local(self, S, etr, tauc, sig, dt):
        gd, slope, pot = self._rates(self.M, sig, tauc, dt)
        for _ in range(80):
            Ss = torch.einsum("vij,vj->vi", S, sig)
            phi = (sig * (0.5 * Ss - etr)).sum(1) + pot
            r = Ss - etr + dt * torch.einsum("vai,va->vi", self.M, gd)
            K = S + dt * torch.einsum("vai,va,vaj->vij", self.M, slope, self.M)
            d = torch.linalg.solve(K, r.unsqueeze(-1)).squeeze(-1)
            rd, dn = (r * d).sum(1), d.norm(dim=1)
            scale = sig.norm(dim=1) + tauc
            step = torch.ones_like(rd)
            for _ in range(40):
                trial = sig - step[:, None] * d
                gd, slope, pot = self._rates(self.M, trial, tauc, dt)
                St = torch.einsum("vij,vj->vi", S, trial)
                bad = ((trial * (0.5 * St - etr)).sum(1) + pot > phi - 1e-4 * step * rd) & (step * dn > 1e-7 * scale)
                if not bool(bad.any()):
                    break
                step = torch.where(bad, 0.5 * step, step)
            sig = trial
            if bool((dn <= 1e-13 * scale).all()):
                break
        return sig

    def _project(self, p):
        """-Gamma0 p (compliance of the reference medium at frequencies with a Nyquist component)."""
        n, r2 = self.n, math.sqrt(2.0)
        f = torch.fft.rfftn(p.T.reshape(6, n, n, n), dim=(1, 2, 3))
        t = torch.empty(f.shape[1:] + (3, 3), dtype=f.dtype, device="cuda")
        for c, (i, j) in enumerate(_PAIRS):
            t[..., i, j] = t[..., j, i] = f[c] / (1.0 if i == j else r2)
        d = self.dir.to(f.dtype)
        v = torch.einsum("...ij,...j->...i", t, d)
        nv = (v * d).sum(-1)
        c = (self.lam0 + self.mu0) / (self.mu0 * (self.lam0 + 2 * self.mu0))
        e = torch.einsum("...i,...j->...ij", d, v)
        e = (e + e.transpose(-1, -2)) / (2 * self.mu0) - c * nv[..., None, None] * d[..., :, None] * d[..., None, :]
        out = -_mandel(e)
        s0 = -torch.einsum("ij,j...->...i", self.S0.to(f.dtype), f)
        out = torch.where(self.nyq[..., None], s0, out)
        out[0, 0, 0] = 0
        return torch.fft.irfftn(out.movedim(-1, 0), s=(n, n, n), dim=(1, 2, 3)).reshape(6, -1).T

    def increment(self, dE33, dt):
        m = self.mat
        tauc = m.tau0 + m.alpha * m.mu * m.b * self.rho.sum(1).sqrt()
        if self.dE is None:
            nu = m.lam / (2 * (m.lam + m.mu))
            dE = np.array([-nu * dE33, -nu * dE33, dE33, 0, 0, 0.0])
            et = self.ee + torch.tensor(dE, device="cuda")
        else:
            dE = self.dE * (dE33 / self.dE[2])
            et = self.ee + self.de * (dE33 / self.dE[2])
        sig = self._local(self.S, et, tauc, self.sig, dt)
        lam, e = sig, et
        C0, S0 = self.C0, self.S0
        uu = [0, 1, 3, 4, 5]
        C0uu = torch.linalg.inv(C0[uu][:, uu]).cpu().numpy()
        for _ in range(2000):
            dE[uu] -= C0uu @ lam.mean(0).cpu().numpy()[uu]
            et = self.ee + torch.tensor(dE, device="cuda") + self._project(lam - (e - self.ee) @ C0)
            ep = et + lam @ S0
            sig = self._local(self.S + S0, ep, tauc, sig, dt)
            e = ep - sig @ S0
            gap = (et - e) @ C0
            lam = lam + gap
            mean = sig.mean(0)
            rms = float(gap.pow(2).sum(1).mean().sqrt() / mean.norm())
            if rms < 1e-11 and float(lam.mean(0)[uu].norm() / mean.norm()) < 1e-11:
                break
        gd, _, _ = self._rates(self.M, sig, tauc, dt)
        dep = dt * torch.einsum("vai,va->vi", self.M, gd)
        self.ep = self.ep + dep
        self.de = et - self.ee
        self.ee = et - dep
        srf = self.rho.sum(1, keepdim=True).sqrt()
        self.rho = self.rho + dt * (m.k1 * srf - m.k2 * self.rho) * gd.abs()
        self.sig, self.dE = sig, dE
        self.E = self.E + dE
        return sig.mean(0)


_EMPTY = 2 ** 30


def _group(ids, vals):
    """Rows of (id, values...) pairs -> per row the distinct ids ascending (_EMPTY last) and the values summed."""
    ids, order = ids.sort(dim=1, stable=True)
    at = torch.cat([torch.zeros_like(ids[:, :1]), (ids[:, 1:] != ids[:, :-1]).long()], 1).cumsum(1)
    out_ids = torch.full_like(ids, _EMPTY).scatter_(1, at, ids)
    return out_ids, [torch.zeros_like(v).scatter_add_(1, at, v.gather(1, order)) for v in vals]


class _PhaseField64:
    """Active-set Allen-Cahn steps, nucleation and statistics in FP64; lists as (points, kmax), _EMPTY = no entry."""

    def __init__(self, case, seed, mat):
        self.n, self.r, self.K, self.G, self.mat = case["n"], case["refine"], case["kmax"], case["grains"], mat
        self.m = self.n * self.r
        rho, self.kappa = _drx_inputs(case, seed, mat)
        self.rho = rho.double()
        self.k = self.rho.sum(0)
        self.t = rho.dtype
        self.g = _voronoi64(self.n, _grains(case, seed)[0])
        up = self.g.reshape(self.n, self.n, self.n)
        for a in range(3):
            up = up.repeat_interleave(self.r, a)
        self.gpf = up.reshape(-1)
        self.ids = torch.full((self.m ** 3, self.K), _EMPTY, dtype=torch.int64, device="cuda")
        self.ids[:, 0] = self.gpf
        self.eta = torch.zeros((self.m ** 3, self.K), dtype=torch.float64, device="cuda")
        self.eta[:, 0] = 1.0
        self.scale = mat.zeta * mat.mu * 1e6 * mat.b ** 2 * (mat.dx / self.r) / mat.omega_gb

    def _kpf(self):
        k = self.k.reshape(self.n, self.n, self.n)
        if self.r == 2:
            for a in range(3):
                lo, hi = 0.25 * k.roll(1, a) + 0.75 * k, 0.75 * k + 0.25 * k.roll(-1, a)
                k = torch.stack([lo, hi], a + 1).flatten(a, a + 1)
        return k.reshape(-1)

    def _shift(self, a, axis, by):
        return a.reshape(self.m, self.m, self.m, -1).roll(by, axis).reshape(self.m ** 3, -1)

    def _sums(self):
        e2 = self.eta ** 2
        D = torch.where(self.ids < self.G, e2, 0.0).sum(1, keepdim=True)
        return D, e2.sum(1, keepdim=True) - D

    def _step(self, kpf):
        mat, K = self.mat, self.K
        m, kap = 6.0 / mat.l_gb, 0.75 * mat.l_gb
        shifts = [(ax, by) for ax in range(3) for by in (1, -1)]
        ids = torch.cat([self.ids] + [self._shift(self.ids, *s) for s in shifts], 1)
        nb = torch.cat([torch.zeros_like(self.eta)] + [self._shift(self.eta, *s) for s in shifts], 1)
        own = torch.zeros_like(nb)
        own[:, :K] = self.eta
        ids, (own, nb) = _group(ids, [own, nb])
        D, R = self._sums()
        S = D + R
        e = 2 * self.scale * kpf[:, None] * own / torch.where(S > 1e-12, S * S, 1.0)
        drive = torch.where(S > 1e-12, torch.where(ids < self.G, e * R, -e * D), 0.0)
        en = own - mat.L_dt * (m * (own ** 3 - own + 3.0 * own * (S - own ** 2)) - kap * (nb - 6 * own) + drive)
        en = torch.where(ids < _EMPTY, en, -math.inf)
        val, at = en.sort(dim=1, descending=True, stable=True)
        val, at = val[:, :K], at[:, :K]
        keep = val >= mat.eta_drop
        keep[:, 0] = True
        kid = torch.where(keep, ids.gather(1, at), _EMPTY)
        self.gpf = kid[:, 0].clone()
        self.ids, order = kid.sort(dim=1)
        self.eta = torch.where(keep, val, 0.0).gather(1, order)

    def steps(self, count):
        before, kpf = self.g, self._kpf()
        for _ in range(count):
            self._step(kpf)
        self.g = self.gpf
        if self.r == 2:
            n = self.n
            kids = lambda a: a.reshape(n, 2, n, 2, n, 2, -1).permute(0, 2, 4, 1, 3, 5, 6).reshape(n ** 3, -1)  # noqa: E731
            ids, (s,) = _group(kids(self.ids), [kids(self.eta)])
            self.g = ids.gather(1, torch.where(ids < _EMPTY, s, -1.0).argmax(1, keepdim=True))[:, 0]
        self._soften((before < self.G) & (self.g >= self.G))

    def _soften(self, sel):
        self.rho = torch.where(sel[None], (self.mat.s_soften * self.rho).to(self.t).double(), self.rho)
        self.k = self.rho.sum(0)

    def nucleate(self):
        g = self.g.reshape(self.n, self.n, self.n)
        gb = torch.zeros_like(g, dtype=torch.bool)
        for ax in range(3):
            for by in (1, -1):
                gb |= g != g.roll(by, ax)
        sel = gb.reshape(-1) & (self.k > self.kappa)
        new = self.G + sel.long().cumsum(0) - 1
        self.g = torch.where(sel, new, self.g)
        self._soften(sel)

        def up(a):
            a = a.reshape(self.n, self.n, self.n)
            for ax in range(3):
                a = a.repeat_interleave(self.r, ax)
            return a.reshape(-1)

        s, i = up(sel), up(new)
        self.ids = torch.where(s[:, None], _EMPTY, self.ids)
        self.eta = torch.where(s[:, None], 0.0, self.eta)
        self.ids[:, 0] = torch.where(s, i, self.ids[:, 0])
        self.eta[:, 0] = torch.where(s, 1.0, self.eta[:, 0])
        self.gpf = torch.where(s, i, self.gpf)

    def energy(self):
        mat, e2 = self.mat, self.eta ** 2
        D, R = self._sums()
        S = (D + R)[:, 0]
        pairs = 0.5 * (S ** 2 - (e2 ** 2).sum(1))
        f0 = 0.25 + (e2 ** 2 / 4 - e2 / 2).sum(1) + 1.5 * pairs
        grad = torch.zeros_like(S)
        for ax in range(3):
            ids, eta = self._shift(self.ids, ax, -1), self._shift(self.eta, ax, -1)
            grad += S + (eta ** 2).sum(1)
            for j in range(self.K):
                hit = (self.ids == ids[:, j:j + 1]) & (self.ids < _EMPTY)
                grad -= 2.0 * (torch.where(hit, self.eta, 0.0) * eta[:, j:j + 1]).sum(1)
        stored = torch.where(S > 1e-12, self.scale * self._kpf() * D[:, 0] / S, 0.0)
        return float((6.0 / mat.l_gb * f0 + 0.375 * mat.l_gb * grad + stored).sum())


def exact(case, seed):
    kind, n = case["kind"], case["n"]
    if kind in ("transform", "residual"):
        x = _fields(case, seed).double()
        if kind == "transform":
            return {"back": x * float(n ** 3)}
        f = torch.fft.rfftn(x, dim=(1, 2, 3))
        k = torch.fft.fftfreq(n, 1.0 / n, dtype=torch.float64, device="cuda")
        k = torch.where(k == -(n // 2), n // 2, k)    # index N/2 counts as +N/2
        full = torch.fft.fftn(x, dim=(1, 2, 3))
        xi = [2 * math.pi / n * a for a in (k[None, None, :], k[None, :, None], k[:, None, None])]
        total = 0.0
        for i in range(3):
            d = sum(xi[j] * full[_PAIRS.index((min(i, j), max(i, j)))] / (1.0 if i == j else math.sqrt(2.0))
                    for j in range(3))
            total += float(d.abs().pow(2).sum())
        return {"spec": f, "out": torch.cat([x.mean(dim=(1, 2, 3)),
                                             torch.tensor([total], dtype=torch.float64, device="cuda")])}
    mat = _material(case)
    if kind == "gradient":
        if n > 16:
            return None   # the curve alone takes about 20 s
        th = _theta(case, seed)
        mech = _Mechanics64(case, seed, dataclasses.replace(mat, **dict(zip(autograd.PARAMS, th.tolist()))))
        curve = [float(mech.increment(*_loading(case))[2]) for _ in range(case["increments"])]
        return {"curve": torch.tensor(curve, dtype=torch.float64), "grad": None}
    if kind == "drx":
        pf = _PhaseField64(case, seed, mat)
        pf.steps(WARM_STEPS)
        pf.nucleate()
        pf.steps(case["steps"])
        return {"ids": None, "eta": pf.eta.T.contiguous(), "g": None, "rho": pf.rho, "k": pf.k[None], "nuclei": None,
                "F_tot": pf.energy(), "X_rex": float((pf.gpf >= pf.G).double().mean()), "n_grains": None,
                "overflow": None}
    if case["law"] == "mr" or n > 32:
        return None   # over 20 s
    mech = _Mechanics64(case, seed, mat)
    for _ in range(case["history"] + 1):
        mean = mech.increment(*_loading(case))
    t = lambda a: a.T.contiguous()  # noqa: E731
    return {"sig": t(mech.sig), "epsp": t(mech.ep), "epse": t(mech.ee), "rho": t(mech.rho), "sig_mean": mean,
            "E": mech.E}
