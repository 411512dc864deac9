"""Performance cases of the phase-field fracture library: what a user's program has it do,
through the public binding (paper_2203_16467_gb300.pff), from the smallest operator call to
a batch of whole load steps.

Kinds of a case:
  laplacian  the allocation-free collocation Laplacian of a device field;
  mechanics  one mechanics sub-problem (Newton-CG) from a given phase field and zero eps*;
  phase      one phase-field sub-problem (BCCG) from a given phase field and strain;
  step       one load step (mechanics, rescale, phase field, post-step) of one simulation, from
             the damage and eps* that the step before left;
  batch      one such load step of several simulations advanced together.
A pass of the solver kinds hands the state in (device tensors), runs the solve and leaves the
new state in the problem's own device fields, which are what it returns.  Grids are powers
of two from 16 to 2048 per side (the library's range), square and not.  Tolerances are the
library's defaults (the paper's).  ``mixed`` problems store FP32 fields, the others FP64.
"""
import ctypes
import math

import numpy as np
import torch

from paper_2203_16467_gb300 import pff
from paper_2203_16467_gb300.inputs import eps_M

NU, GC = 0.2, 1.0


# ------------------------------------------------------------------------------ the cases
def listed():
    return [
        # the smallest call: one operator on a 64^2 field inside somebody else's loop (latency)
        {"name": "laplacian_f32_64", "kind": "laplacian", "nx": 64, "ny": 64, "mixed": True},
        # the same operator in FP64 on a non-square grid
        {"name": "laplacian_f64_512x256", "kind": "laplacian", "nx": 512, "ny": 256, "mixed": False},
        # the mechanics of the 64^2 crack-path workload: many short iterations
        {"name": "mechanics_64", "kind": "mechanics", "nx": 64, "ny": 64, "mixed": True, "fracture": "AT1",
         "split": "SPECTRAL", "irreversibility": "CRACK_SET", "ell": 2.0, "load": 1.1},
        # an FP64 reference solve on a non-square grid, isotropic contact (a linear solve)
        {"name": "mechanics_f64_256x128", "kind": "mechanics", "nx": 256, "ny": 128, "mixed": False,
         "fracture": "AT1", "split": "ISOTROPIC", "irreversibility": "CRACK_SET", "ell": 2.0, "load": 1.0},
        # the mechanics of one simulation of the four-way model comparison's grid
        {"name": "mechanics_512", "kind": "mechanics", "nx": 512, "ny": 512, "mixed": True, "fracture": "AT2",
         "split": "SPECTRAL", "irreversibility": "CRACK_SET", "ell": 4.0, "load": 1.0},
        # a small non-square phase-field solve (a specimen strip)
        {"name": "phase_128x64", "kind": "phase", "nx": 128, "ny": 64, "mixed": True, "fracture": "AT1",
         "split": "SPECTRAL", "irreversibility": "CRACK_SET", "ell": 2.0, "load": 1.2},
        # the phase-field solve of one simulation of the four-way model comparison's grid
        {"name": "phase_512", "kind": "phase", "nx": 512, "ny": 512, "mixed": True, "fracture": "AT2",
         "split": "SPECTRAL", "irreversibility": "DAMAGE", "ell": 4.0, "load": 1.1},
        # an FP64 reference phase-field solve
        {"name": "phase_f64_256", "kind": "phase", "nx": 256, "ny": 256, "mixed": False, "fracture": "AT1",
         "split": "ISOTROPIC", "irreversibility": "DAMAGE", "ell": 2.0, "load": 1.1},
        # one load step of the 64^2 crack-path workload (a whole run takes several hundred)
        {"name": "step_64", "kind": "step", "nx": 64, "ny": 64, "mixed": True, "fracture": "AT1",
         "split": "SPECTRAL", "irreversibility": "CRACK_SET", "ell": 2.0, "load": 1.05},
        # one load step of the largest grid
        {"name": "step_2048", "kind": "step", "nx": 2048, "ny": 2048, "mixed": True, "fracture": "AT2",
         "split": "SPECTRAL", "irreversibility": "CRACK_SET", "ell": 2.0, "load": 0.97},
        # the benchmark's batch: eight model variants on one microstructure, a stream each
        {"name": "batch8_512", "kind": "batch", "nx": 512, "ny": 512, "mixed": True, "members": 8, "group": 1,
         "fracture": "ALL", "split": "ALL", "irreversibility": "ALL", "ell": 4.0, "load": 0.97},
        # an ensemble of microstructures under one model, in lock-step groups of eight
        {"name": "batch64_256", "kind": "batch", "nx": 256, "ny": 256, "mixed": True, "members": 64, "group": 8,
         "fracture": "AT1", "split": "SPECTRAL", "irreversibility": "CRACK_SET", "ell": 2.0, "load": 1.0},
    ]


def _pow2(rng, lo, hi):
    return 2 ** rng.randint(int(math.log2(lo)), int(math.log2(hi)))


def draw(rng):
    """Any kind, any grid of its range, any model; FP64 solves up to 2^17 pixels, mixed ones up to
    2^22 (single) and 2^21 (a batch's sum, its members up to 512 a side)."""
    kind = rng.choice(["laplacian", "mechanics", "mechanics", "phase", "phase", "step", "step", "batch"])
    mixed = rng.random() < 0.7
    if kind == "laplacian":
        return {"kind": kind, "nx": _pow2(rng, 16, 512), "ny": _pow2(rng, 16, 512), "mixed": mixed}
    case = {"kind": kind, "mixed": mixed, "fracture": rng.choice(["AT1", "AT2"]),
            "split": rng.choice(["ISOTROPIC", "SPECTRAL", "SPECTRAL", "VOLDEV"]),
            "irreversibility": rng.choice(["CRACK_SET", "DAMAGE"]),
            "ell": round(rng.uniform(1.5, 4.0), 3), "load": round(rng.uniform(0.9, 1.2), 4)}
    side = 512 if kind == "batch" else 2048
    while True:
        nx, ny = _pow2(rng, 16, side), _pow2(rng, 16, side)
        if max(nx, ny) <= 16 * min(nx, ny) and nx * ny <= (2 ** 22 if mixed else 2 ** 17):
            break
    case.update(nx=nx, ny=ny)
    if kind == "batch":
        most = min(32, 2 ** (21 if mixed else 18) // (nx * ny))
        case["members"] = rng.randint(2, max(2, most))
        case["group"] = rng.choice([1, 4, 8, 0])
    return case


# ------------------------------------------------------------------------------ inputs
def _smooth(nx, ny, lc, gen, lead=()):
    """Gaussian random fields of correlation length lc (pixels), zero mean and unit variance."""
    w = torch.randn(*lead, ny, nx, dtype=torch.float64, device="cuda", generator=gen)
    qy = torch.fft.fftfreq(ny, dtype=torch.float64, device="cuda")[:, None]
    qx = torch.fft.rfftfreq(nx, dtype=torch.float64, device="cuda")[None, :]
    f = torch.exp(-(2.0 * math.pi) ** 2 * (qx * qx + qy * qy) * lc * lc / 4.0)
    z = torch.fft.irfft2(torch.fft.rfft2(w) * f, s=(ny, nx))
    z = z - z.mean(dim=(-2, -1), keepdim=True)
    return z / z.std(dim=(-2, -1), keepdim=True)


def _store(t, mixed):
    """Values as the problem stores them (FP32 for mixed), handed over as FP64."""
    return (t.float().double() if mixed else t).contiguous()


def _inputs(case, seed):
    """Modulus, phase field, eps*, eps_bar of every simulation of a case, from the seed."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    nx, ny, mixed = case["nx"], case["ny"], case["mixed"]
    m = case.get("members", 1)
    same = case["fracture"] == "ALL"          # the model variants share one microstructure
    n = min(nx, ny)
    z = _smooth(nx, ny, max(2.0, n / 16.0), gen, (1 if same else m,))
    E = torch.exp(0.3 * z)
    E = _store(E / E.mean(dim=(-2, -1), keepdim=True), mixed)
    E = E.expand(m, ny, nx).contiguous()
    bumps = _smooth(nx, ny, 4.0 if n >= 32 else 2.0, gen, (m,))
    lo, hi = bumps.amin(dim=(-2, -1), keepdim=True), bumps.amax(dim=(-2, -1), keepdim=True)
    top = {"mechanics": 0.8, "phase": 0.95, "step": 0.3, "batch": 0.3}[case["kind"]]
    # damage concentrated in a few places, as along cracks
    phi = _store(top * ((bumps - lo) / (hi - lo)) ** 3, mixed)
    em = eps_M(1.0, NU, GC, case["ell"])
    eps_bar, eps_star = (0.0, case["load"] * em, 0.0), None
    if case["kind"] == "mechanics":
        return E, phi, [None] * m, eps_bar, em
    # the state that the step before left: damage near equilibrium under a twentieth of eps_M less
    before = (0.0, (case["load"] - 0.05) * em, 0.0)
    phis, stars = [], []
    for j, (f, sp, ir) in enumerate(_models(case)):
        model = _Model(dict(case, fracture=f, split=sp, irreversibility=ir), E[j], case["ell"])
        if case["kind"] == "phase":           # any strained, inhomogeneous state
            e = _smooth(nx, ny, 4.0 if n >= 32 else 2.0, gen, (3,))
            star = 0.3 * em * (e - e.mean(dim=(-2, -1), keepdim=True))
            strain = (1.0 - 0.05 / case["load"]) * (model.bar(eps_bar) + star)
        else:
            star = model.mechanics(phi[j], before, 1e-3)
            strain = model.bar(before) + star
        phis.append(_store(model.phase(phi[j], strain, 1e-3, 60), mixed))
        stars.append(_store(star, mixed))
    return E, torch.stack(phis), stars, eps_bar, em


MODELS8 = [(f, s, i) for f in ("AT1", "AT2") for s in ("ISOTROPIC", "SPECTRAL") for i in ("CRACK_SET", "DAMAGE")]


def _models(case):
    if case["fracture"] == "ALL":
        return [MODELS8[j % 8] for j in range(case["members"])]
    return [(case["fracture"], case["split"], case["irreversibility"])] * case.get("members", 1)


class _Device:
    """Array interface of a device field that a problem holds (and that keeps the problem alive)."""

    def __init__(self, problem, ptr, shape, dtype):
        self.problem = problem
        self.__cuda_array_interface__ = {"data": (ptr, False), "shape": shape, "typestr": "<f4" if dtype else "<f8",
                                         "version": 2, "strides": None}


def _view(problem, which, ncomp):
    ptr, dtype = problem.get_device_ptr(which)
    shape = (ncomp, problem.ny, problem.nx) if ncomp > 1 else (problem.ny, problem.nx)
    return torch.as_tensor(_Device(problem, ptr, shape, dtype), device="cuda")


class State:
    batch = None

    def __del__(self):
        if self.batch is not None:
            pff.destroy_batch(self.batch)
            self.batch = None


def prepare(case, seed):
    s = State()
    s.kind = case["kind"]
    nx, ny, mixed = case["nx"], case["ny"], case["mixed"]
    if s.kind == "laplacian":
        gen = torch.Generator(device="cuda")
        gen.manual_seed(int(seed))
        t = torch.float32 if mixed else torch.float64
        s.src = (_smooth(nx, ny, max(2.0, nx / 16.0), gen) + 0.3 * torch.randn(
            ny, nx, dtype=torch.float64, device="cuda", generator=gen)).to(t)
        s.dst = torch.empty_like(s.src)
        s.fn = pff.lib.pff_apply_laplacian_noalloc_f32 if mixed else pff.lib.pff_apply_laplacian_noalloc
        # on the caller's stream: calls share the library's scratch, so they are serialised
        s.args = (nx, ny, 1.0, ctypes.c_void_p(s.src.data_ptr()), ctypes.c_void_p(s.dst.data_ptr()),
                  ctypes.c_void_p(torch.cuda.current_stream().cuda_stream), None)
        torch.cuda.synchronize()
        return s
    E, s.phi, s.eps_star, s.eps_bar, em = _inputs(case, seed)
    s.stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    prec = pff.MIXED if mixed else pff.FP64
    s.problems = [pff.Problem(nx, ny, prec, stream=s.stream.cuda_stream, E=E[j], model=model,
                              params=dict(nu=NU, Gc=GC, ell=case["ell"], d_eps_bar=(0.0, em / 20.0, 0.0)))
                  for j, model in enumerate(_models(case))]
    if s.kind == "batch":
        m = case["members"]
        s.batch = pff.create_batch(m, m * pff.problem_bytes(nx, ny, prec), s.stream.cuda_stream)
        for p in s.problems:
            pff.batch_admit(s.batch, p.h)
        pff.batch_set_group_size(s.batch, case["group"])
    s.phi_out = [_view(p, pff.FIELD_PHI, 1) for p in s.problems]
    s.eps_out = [_view(p, pff.FIELD_EPS_STAR, 3) for p in s.problems]
    torch.cuda.synchronize()
    return s


def run(state):
    s = state
    if s.kind == "laplacian":
        rc = s.fn(*s.args)
        if rc:
            raise RuntimeError(f"laplacian: error {rc}")
        return s.dst
    for j, p in enumerate(s.problems):
        p.set_phase_field(s.phi[j])
        p.set_strain(s.eps_star[j], s.eps_bar)
    if s.kind == "mechanics":
        s.problems[0].solve_mechanics()
        return s.eps_out[0]
    if s.kind == "phase":
        s.problems[0].solve_phase_field()
        return s.phi_out[0]
    for p in s.problems:
        p.set_flag(0)
    if s.kind == "step":
        r = s.problems[0].step_load(1)[0]
        return {"phi": s.phi_out[0], "eps_star": s.eps_out[0], "eps_bar": r["eps_bar"], "sig_bar": r["sig_bar"],
                "C_bar": r["C_bar"], "F_e": r["F_e"], "F_f": r["F_f"]}
    reps = pff.batch_step(s.batch, len(s.problems), 1)
    with torch.cuda.stream(s.stream):         # the problems' own stream: before its next state comes in
        phi, eps_star = torch.stack(s.phi_out), torch.stack(s.eps_out)
    return {"phi": phi, "eps_star": eps_star,
            "sig_bar": np.array([r[0]["sig_bar"] for r in reps], dtype=np.float32)}


# ------------------------------------------------------------------------------ work
def work(case):
    """Inputs read and outputs written once; operations of the transforms and pointwise work at
    iteration counts typical of the kind (the solves stop by tolerance, not by count)."""
    n = case["nx"] * case["ny"]
    es = 4 if case["mixed"] else 8
    fft = 2.5 * n * math.log2(n)                     # one real 2-D transform
    if case["kind"] == "laplacian":
        return {"bytes": 2 * n * es, "flops": 2 * fft + 2 * n}
    cg, pf = 6 * fft + 120 * n, 2 * fft + 40 * n     # one iteration of either solver
    m = case.get("members", 1)
    its = {"mechanics": (60, 0), "phase": (0, 80), "step": (30, 80), "batch": (30, 80)}[case["kind"]]
    # handed in: phi and (but for mechanics) eps* in FP64; held: E; written: phi and / or eps*
    words = {"mechanics": 8 + 4 * es, "phase": 4 * 8 + 2 * es, "step": 4 * 8 + 5 * es, "batch": 4 * 8 + 5 * es}
    return {"bytes": m * n * words[case["kind"]], "flops": m * (its[0] * cg + its[1] * pf)}


# ------------------------------------------------------------------------------ 64-bit values
def _pos(x):
    return torch.clamp(x, min=0.0)


class _Model:
    """Plain FP64 torch statement of the sub-problems (2-D plane strain, planes xx, yy, xy)."""

    def __init__(self, case, E, ell):
        self.nx, self.ny = case["nx"], case["ny"]
        self.at1, self.split = case["fracture"] == "AT1", case["split"]
        self.damage = case["irreversibility"] == "DAMAGE"
        self.lam, self.mu = E * NU / ((1 + NU) * (1 - 2 * NU)), E / (2 * (1 + NU))
        self.c = GC / ((8.0 / 3.0 if self.at1 else 2.0) * ell)
        self.ell, self.kappa = ell, 2 * self.c * ell * ell
        self.eta_dt = 2.0 ** -16 * GC / ell
        dev = dict(dtype=torch.float64, device=E.device)
        qx = 2 * math.pi * torch.fft.rfftfreq(self.nx, **dev)[None, :]
        qy = 2 * math.pi * torch.fft.fftfreq(self.ny, **dev)[:, None]
        self.q2 = qx * qx + qy * qy
        inv = torch.rsqrt(torch.where(self.q2 > 0, self.q2, torch.ones_like(self.q2)))
        keep = (self.q2 > 0).double()
        keep[:, self.nx // 2] = 0
        keep[self.ny // 2, :] = 0
        self.n1, self.n2, self.keep = qx * inv, qy * inv, keep

    def bar(self, eps_bar):
        return torch.tensor(eps_bar, dtype=torch.float64, device=self.lam.device)[:, None, None]

    def lap(self, f):
        return torch.fft.irfft2(-self.q2 * torch.fft.rfft2(f), s=(self.ny, self.nx))

    def project(self, z):
        a, b, c = torch.fft.rfft2(z)
        n1, n2 = self.n1, self.n2
        s1, s2 = n1 * a + n2 * c, n1 * c + n2 * b
        t = n1 * s1 + n2 * s2
        g = torch.stack([2 * n1 * s1 - t * n1 * n1, 2 * n2 * s2 - t * n2 * n2, n1 * s2 + n2 * s1 - t * n1 * n2])
        return torch.fft.irfft2(g * self.keep, s=(self.ny, self.nx))

    def _eig(self, e):
        d, tr = 0.5 * (e[0] - e[1]), e[0] + e[1]
        rad = torch.sqrt(d * d + e[2] * e[2])
        ir = torch.where(rad > 0, 1 / rad.clamp(min=1e-300), torch.zeros_like(rad))
        u = torch.where(rad > 0, d * ir, torch.ones_like(rad))
        return tr, 0.5 * tr + rad, 0.5 * tr - rad, u, e[2] * ir, rad

    def psi(self, e):
        tr, lam, mu = e[0] + e[1], self.lam, self.mu
        if self.split == "ISOTROPIC":
            return 0.5 * lam * tr ** 2 + mu * (e[0] ** 2 + e[1] ** 2 + 2 * e[2] ** 2)
        if self.split == "VOLDEV":
            K, a, b = lam + 2 * mu / 3, e[0] - tr / 3, e[1] - tr / 3
            return 0.5 * K * _pos(tr) ** 2 + mu * (a * a + b * b + 2 * e[2] ** 2)
        tr, e1, e2, _, _, _ = self._eig(e)
        return 0.5 * lam * _pos(tr) ** 2 + mu * (_pos(e1) ** 2 + _pos(e2) ** 2)

    def energy(self, e, h):
        tr, lam, mu = e[0] + e[1], self.lam, self.mu
        if self.split == "ISOTROPIC":
            return h * self.psi(e)
        if self.split == "VOLDEV":
            return h * self.psi(e) + 0.5 * (lam + 2 * mu / 3) * _pos(-tr) ** 2
        tr, e1, e2, _, _, _ = self._eig(e)
        return h * self.psi(e) + 0.5 * lam * _pos(-tr) ** 2 + mu * (_pos(-e1) ** 2 + _pos(-e2) ** 2)

    def stress(self, e, h):
        lam, mu, tr = self.lam, self.mu, e[0] + e[1]
        one = torch.stack([torch.ones_like(tr), torch.ones_like(tr), torch.zeros_like(tr)])
        if self.split == "ISOTROPIC":
            return h * (lam * tr * one + 2 * mu * e)
        if self.split == "VOLDEV":
            K = lam + 2 * mu / 3
            return h * (K * _pos(tr) * one + 2 * mu * (e - 4.0 / 9.0 * tr * one)) - K * _pos(-tr) * one
        tr, e1, e2, u, w, _ = self._eig(e)
        a1, a2 = _pos(e1), _pos(e2)
        hs, hd = 0.5 * (a1 + a2), 0.5 * (a1 - a2)
        ep = torch.stack([hs + hd * u, hs - hd * u, hd * w])
        return h * (lam * _pos(tr) * one + 2 * mu * ep) - lam * _pos(-tr) * one + 2 * mu * (e - ep)

    def tangent(self, e, h):
        lam, mu, tr = self.lam, self.mu, e[0] + e[1]
        one = torch.stack([torch.ones_like(tr), torch.ones_like(tr), torch.zeros_like(tr)])
        Ht = (tr > 0).double()
        if self.split == "ISOTROPIC":
            return lambda p: h * (lam * (p[0] + p[1]) * one + 2 * mu * p)
        if self.split == "VOLDEV":
            K = lam + 2 * mu / 3
            return lambda p: (h * (K * Ht * (p[0] + p[1]) * one + 2 * mu * (p - 4.0 / 9.0 * (p[0] + p[1]) * one))
                              + K * (1 - Ht) * (p[0] + p[1]) * one)
        tr, e1, e2, u, w, rad = self._eig(e)
        H1, H2 = (e1 > 0).double(), (e2 > 0).double()
        g = torch.where(rad > 0, (_pos(e1) - _pos(e2)) / (2 * rad).clamp(min=1e-300), H1)

        def apply(p):
            t = p[0] + p[1]
            P1 = 0.5 * ((1 + u) * p[0] + (1 - u) * p[1] + 2 * w * p[2])
            P2 = t - P1
            S = 0.5 * (-w * p[0] + w * p[1] + 2 * u * p[2])
            c1, c2, c3 = H1 * P1, H2 * P2, g * S
            D = torch.stack([0.5 * (c1 * (1 + u) + c2 * (1 - u)) - c3 * w,
                             0.5 * (c1 * (1 - u) + c2 * (1 + u)) + c3 * w, 0.5 * (c1 - c2) * w + c3 * u])
            return h * (lam * Ht * t * one + 2 * mu * D) + lam * (1 - Ht) * t * one + 2 * mu * (p - D)
        return apply

    @staticmethod
    def dot(a, b):
        return float((a[0] * b[0] + a[1] * b[1] + 2 * a[2] * b[2]).sum())

    def mechanics(self, phi, eps_bar, tol=1e-11, start=None):
        bar = self.bar(eps_bar)
        h, e = (1 - phi) ** 2, bar.repeat(1, self.ny, self.nx)
        ref = math.sqrt(self.dot(*[self.stress(e, torch.ones_like(phi))] * 2))
        if start is not None:
            e = e + start
        for _ in range(60):
            r = -self.project(self.stress(e, h))
            rr = self.dot(r, r)
            if math.sqrt(rr) <= tol * ref:
                break
            stop, C = max(1e-4 * math.sqrt(rr), 0.3 * tol * ref), self.tangent(e, h)
            x, p = torch.zeros_like(r), r.clone()
            for _ in range(4000):
                q = self.project(C(p))
                a = rr / self.dot(p, q)
                x += a * p
                r -= a * q
                new = self.dot(r, r)
                if math.sqrt(new) <= stop:
                    break
                p = r + new / rr * p
                rr = new
            e = e + x
        return e - bar

    def phase(self, phi, e, tol=1e-12, most=6000):
        psi, lap = self.psi(e), self.lap(phi)
        a = self.eta_dt + 2 * psi + (0.0 if self.at1 else 2 * self.c)
        b = 2 * (1 - phi) * psi - self.c * (torch.ones_like(phi) if self.at1 else 2 * phi) + self.kappa * lap
        con = phi if self.damage else torch.where(phi >= 0.9, phi, torch.zeros_like(phi))
        low = con - phi
        J = lambda x: a * x - self.kappa * self.lap(x)  # noqa: E731
        v = torch.maximum(torch.zeros_like(phi), low)
        r = J(v) - b
        r[(v == low) & (r > 0)] = 0.0
        p, stop = -r, tol * float(r.norm())
        for _ in range(most):
            Jp = J(p)
            pJp = float((p * Jp).sum())
            if pJp <= 0:
                break
            al = -float((r * p).sum()) / pJp
            v = torch.maximum(v + al * p, low)
            old, r = r, J(v) - b
            act = (v == low) & (r > 0)
            r[act] = 0.0
            if float(r.norm()) <= stop:
                break
            p = -r + float((r * (r - old)).sum()) / (al * pJp) * p
            p[act] = 0.0
        return phi + v

    def step(self, phi, start, eps_bar, d_eps):
        """One load step from the state (phi, eps*, eps_bar, no earlier rescale)."""
        bar = self.bar(eps_bar)
        es = self.mechanics(phi, eps_bar, start=start)
        psi = self.psi(bar + es)
        D = 2 * (1 - phi) * psi
        R = -self.c * (torch.ones_like(phi) if self.at1 else 2 * phi) + self.kappa * self.lap(phi)
        i = int(torch.argmax(D + R))
        top, g = float((D + R).reshape(-1)[i]), 1.0
        fmax = 0.7 * GC / self.ell
        if top > fmax and float(D.max()) > GC / self.ell:
            num, den = fmax - float(R.reshape(-1)[i]), float(D.reshape(-1)[i])
            if num > 0 and den > 0:
                g = min(math.sqrt(num / den), 1 + max(map(abs, d_eps)) / max(map(abs, eps_bar)))
        es, bar = g * es, g * bar
        new = self.phase(phi, bar + es)
        h = (1 - new) ** 2
        sig = self.stress(bar + es, h).mean(dim=(-2, -1)).tolist()
        eb = bar.reshape(3).tolist()
        f = new if self.at1 else new * new
        Ff = self.c * float((f - self.ell ** 2 * new * self.lap(new)).sum())
        return {"phi": new, "eps_star": es, "eps_bar": eb, "sig_bar": sig, "C_bar": sig[1] / eb[1],
                "F_e": float(self.energy(bar + es, h).sum()), "F_f": Ff}


def exact(case, seed):
    if case["kind"] == "laplacian":
        s = prepare(case, seed)
        f = s.src.double()
        qx = 2 * math.pi * torch.fft.rfftfreq(case["nx"], dtype=torch.float64, device="cuda")[None, :]
        qy = 2 * math.pi * torch.fft.fftfreq(case["ny"], dtype=torch.float64, device="cuda")[:, None]
        return torch.fft.irfft2(-(qx * qx + qy * qy) * torch.fft.rfft2(f), s=f.shape)
    if case["kind"] == "batch" or case["nx"] * case["ny"] > 2 ** 19:
        return None                                   # too long
    E, phi, eps_star, eps_bar, em = _inputs(case, seed)
    m = _Model(case, E[0], case["ell"])
    if case["kind"] == "mechanics":
        return m.mechanics(phi[0], eps_bar)
    if case["kind"] == "phase":
        return m.phase(phi[0], m.bar(eps_bar) + eps_star[0])
    r = m.step(phi[0], eps_star[0], eps_bar, (0.0, em / 20.0, 0.0))
    # the values of a report are told as single numbers: FP64 there too
    return {k: ([np.float64(x) for x in v] if isinstance(v, list) else np.float64(v) if isinstance(v, float) else v)
            for k, v in r.items()}
