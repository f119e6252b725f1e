"""What a user of this framework has it do, as cases that can be timed and checked.

A user couples stiff chemistry to a flow solver.  Per time step the solver hands
over every cell's state (mass fractions and temperature) and gets it back
reacted: ``rok4e_integrate`` over independent cells, or ``simpler_split_step``
over the points of a 1-D flame.  Others call the source term or its
Jacobian-vector product inside an integrator of their own, or differentiate a
run of fixed steps with respect to the rate constants.  The mechanisms are the
four of ``synth.fields.WORKLOADS``; states are drawn like their fields.

``listed`` gives the cases, ``draw`` more of the same ranges, ``prepare`` the
tensors and handles a program holds before the call, ``run`` one pass through
the public calls, ``work`` what a pass cannot do without, ``exact`` the same
results from plain float64 torch.
"""

from __future__ import annotations

import functools
import math

import numpy as np
import torch

import paper_1712_00953_gb300 as rk
from synth.fields import P_ATM, WORKLOADS, mechanism_for

RTOL, ATOL = 1e-6, 1e-10  # the tolerances of every workload
D_DIFF, LENGTH = 1.0e-4, 1.0e-2  # the flame's diffusivity (m^2/s) and domain (m)


def listed():
    return [
        # a source term on the 256 cells of the 10-species workload: the smallest call, all latency
        {"name": "rhs_small", "kind": "rhs", "mech": "small", "cells": 256},
        # a source term on a large block of cells at the size of GRI-3.0
        {"name": "rhs_large", "kind": "rhs", "mech": "batched", "cells": 131072},
        # Jacobian-vector products with third-body and Troe reactions, an odd number of cells
        {"name": "jvp_pressure", "kind": "jvp", "mech": "flame1d", "cells": 20011},
        # one reaction step of the 10-species workload: 256 cells do not fill the chip
        {"name": "step_small", "kind": "rok4e", "mech": "small", "cells": 256, "dt": 1e-6, "M": 4, "steps": 1,
         "precision": 0, "volume": False},
        # constant-volume cells (a closed reactor), two time steps with carried step sizes
        {"name": "step_volume", "kind": "rok4e", "mech": "small", "cells": 20001, "dt": 1e-6, "M": 4, "steps": 2,
         "precision": 0, "volume": True},
        # the main path: cells of very uneven stiffness, two time steps with carried step sizes
        {"name": "step_large", "kind": "rok4e", "mech": "batched", "cells": 12288, "dt": 1e-6, "M": 4, "steps": 2,
         "precision": 0, "volume": False},
        # the same in mixed precision (FP32 Jacobian-vector products)
        {"name": "step_mixed", "kind": "rok4e", "mech": "batched", "cells": 6000, "dt": 1e-6, "M": 4, "steps": 2,
         "precision": 6, "volume": False},
        # a larger Krylov space on the mechanism with third-body and Troe reactions, ragged size
        {"name": "step_krylov6", "kind": "rok4e", "mech": "flame1d", "cells": 3001, "dt": 1e-6, "M": 6, "steps": 1,
         "precision": 0, "volume": False},
        # the explicit integrator of non-stiff users and of the efficiency study
        {"name": "explicit", "kind": "rkdp", "mech": "batched", "cells": 8192, "dt": 1e-7, "steps": 2},
        # four split steps of the 2048-point flame from its initial front
        {"name": "flame", "kind": "split", "mech": "flame1d", "cells": 2048, "dt": 1e-7, "M": 4, "steps": 4},
        # a training step: fixed steps with checkpoints, then the gradient by ln A and by the initial state
        {"name": "gradient", "kind": "adjoint", "mech": "adjoint", "cells": 1024, "h": 2e-8, "M": 4, "steps": 10},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["rhs", "jvp", "rok4e", "rok4e", "rok4e", "rkdp", "split", "adjoint"])
    if kind in ("rhs", "jvp"):
        return {"kind": kind, "mech": rng.choice(["small", "flame1d", "batched"]), "cells": _log_int(rng, 100, 100000)}
    if kind == "rok4e":
        mech, top = rng.choice([("small", 30000), ("flame1d", 8000), ("batched", 10000)])
        return {"kind": kind, "mech": mech, "cells": _log_int(rng, 100, top), "dt": 10.0 ** rng.uniform(-7.0, -6.0),
                "M": rng.choice([4, 4, 4, 5, 6]), "steps": rng.choice([1, 2]), "precision": rng.choice([0, 0, 0, 6]),
                "volume": rng.random() < 0.25}
    if kind == "rkdp":
        return {"kind": kind, "mech": rng.choice(["small", "flame1d", "batched"]), "cells": _log_int(rng, 100, 8000),
                "dt": 10.0 ** rng.uniform(-8.0, -7.0), "steps": 2}
    if kind == "split":
        return {"kind": kind, "mech": "flame1d", "cells": _log_int(rng, 100, 2048), "dt": 10.0 ** rng.uniform(-8.0, -7.0),
                "M": 4, "steps": rng.choice([2, 3, 4])}
    return {"kind": kind, "mech": rng.choice(["small", "flame1d", "adjoint"]), "cells": _log_int(rng, 64, 1000),
            "h": 10.0 ** rng.uniform(-8.5, -7.7), "M": 4, "steps": rng.randint(2, 10)}


@functools.lru_cache(maxsize=None)
def _mechanism(name):
    """The mechanism's description on the host, which a program reads once from its file."""
    return mechanism_for(WORKLOADS[name])


def _state(case, seed):
    """Rows (Y, T): Dirichlet(0.5) mass fractions (normalised squares of normals) and the
    workload's temperatures, on the GPU; the flame's front in place of them for a split step."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    ns, n = WORKLOADS[case["mech"]].n_species, case["cells"]

    def dirichlet(rows):
        z = torch.randn(rows, ns, dtype=torch.float64, device="cuda", generator=g).square_()
        return z / z.sum(1, keepdim=True)

    if case["kind"] == "split":
        x = (torch.arange(n, dtype=torch.float64, device="cuda") + 0.5) * (LENGTH / n)
        front = torch.tanh((x - 0.5 * LENGTH) / 1e-3)
        w = (0.5 * (1.0 + front))[:, None]
        return torch.cat([(1.0 - w) * dirichlet(1) + w * dirichlet(1), (1150.0 + 850.0 * front)[:, None]], 1)
    Y = dirichlet(n)
    if case["mech"] in ("small", "adjoint"):
        T = 1000.0 + 500.0 * torch.rand(n, 1, dtype=torch.float64, device="cuda", generator=g)
    else:
        T = torch.randn(n, 1, dtype=torch.float64, device="cuda", generator=g).mul_(300.0).add_(1400.0)
        T.clamp_(300.0, 3000.0 if case["mech"] == "batched" else 2000.0)
    return torch.cat([Y, T], 1)


def _rho(case, U):
    """Densities at 1 atm of the given states: the closed reactors' constants."""
    invW = torch.as_tensor(1.0 / _mechanism(case["mech"]).W, device=U.device)
    return P_ATM / (8.314462618 * U[:, -1] * (U[:, :-1] @ invW))


def _direction(U, seed):
    """The vectors V of the Jacobian-vector products: both signs, temperature entries of order 1."""
    g = torch.Generator(device="cuda").manual_seed(seed + 7919)
    return torch.randn(U.shape, dtype=torch.float64, device="cuda", generator=g)


def _cotangent(case, U):
    """dL/du(t_end) of the loss "sum of final temperatures plus a little of every mass fraction"."""
    w = torch.linspace(0.5, 1.5, U.shape[1], dtype=torch.float64, device=U.device).expand_as(U).clone()
    w[:, -1] = 1.0
    return w


def prepare(case, seed):
    U = _state(case, seed)
    s = {"case": case, "U0": U}
    if case["kind"] == "adjoint":
        d = _mechanism(case["mech"])
        s["mech"] = d
        s["lnA"] = torch.from_numpy(np.log(d.arrh[:, 0])).requires_grad_(True)
        s["w"] = _cotangent(case, U)
        s["U0"] = U.requires_grad_(True)
        return s
    m = s["m"] = rk.mech_load(_mechanism(case["mech"]))
    n = case["cells"]
    if case["kind"] == "jvp":
        s["V"] = _direction(U, seed)
    if case["kind"] in ("rhs", "jvp"):
        s["out"] = torch.empty_like(U)
        return s
    s["U"] = torch.empty_like(U)
    s["h"] = torch.zeros(n, dtype=torch.float64, device="cuda")
    s["stats"] = torch.zeros(n, 4, dtype=torch.int32, device="cuda")
    if case["kind"] == "split":
        s["opts"] = rk.Opts()
        nb = rk.simpler_split_step_workspace_size(m, n, case["M"], s["opts"])
    else:
        s["opts"] = rk.Opts(precision=case.get("precision", 0), rho_cell=_rho(case, U) if case.get("volume") else None)
        nb = rk.rok4e_workspace_size(m, n, case.get("M", 1), s["opts"])
    s["ws"] = torch.empty(nb, dtype=torch.uint8, device="cuda")
    return s


def run(s):
    """One pass.  Time stepping returns the state; the carried step and the counts of attempts that
    the calls also keep are hints and diagnostics whose last digits are rounding of the error estimate."""
    c = s["case"]
    kind = c["kind"]
    if kind == "rhs":
        return rk.chem_rhs(s["m"], s["U0"], P_ATM, out=s["out"])
    if kind == "jvp":
        return rk.chem_jvp(s["m"], s["U0"], s["V"], P_ATM, out=s["out"])
    if kind == "adjoint":
        U = rk.FixedStepROK4E.apply(s["lnA"], s["U0"], s["mech"], c["h"], c["steps"], c["M"], P_ATM)
        g_lnA, g_u0 = torch.autograd.grad((U * s["w"]).sum(), (s["lnA"], s["U0"]))
        return {"U": U.detach(), "g_lnA": g_lnA, "g_u0": g_u0}
    U, h = s["U"], s["h"]
    U.copy_(s["U0"])
    h.zero_()
    for _ in range(c["steps"]):
        kw = dict(h_cell=h, opts=s["opts"], stats=s["stats"], workspace=s["ws"])
        if kind == "split":
            rk.simpler_split_step(s["m"], U, c["dt"], D_DIFF, LENGTH / c["cells"], RTOL, ATOL, c["M"], **kw)
        elif kind == "rkdp":
            rk.rkdp_integrate(s["m"], U, c["dt"], RTOL, ATOL, **kw)
        else:
            rk.rok4e_integrate(s["m"], U, c["dt"], RTOL, ATOL, c["M"], **kw)
    return U


def work(case):
    """States in and out, and floating point operations of the method: per right-hand side 16 a
    reaction, 40 a species and 20 an exponential (one a reaction, two a species), 2 a stoichiometric
    coefficient (four a reaction); a Jacobian-vector product 26 and 25; an attempt of the integrator
    three right-hand sides, M products and its vectors, with the attempts per cell that the method
    takes on these fields (in proportion to dt)."""
    w = WORKLOADS[case["mech"]]
    ns, nr, n, N = w.n_species, w.n_reactions, case["cells"], w.n_species + 1
    rhs = 40 * ns + 16 * nr + 8 * nr + 20 * (2 * ns + nr) + (w.n_third_body + w.n_troe) * 2 * ns
    jvp = 25 * ns + 26 * nr + 8 * nr
    kind, M = case["kind"], case.get("M", 4)
    if kind == "rhs":
        return {"bytes": 16.0 * n * N, "flops": float(n * rhs)}
    if kind == "jvp":
        return {"bytes": 24.0 * n * N, "flops": float(n * (rhs + jvp))}
    attempt = 3 * rhs + M * jvp + N * (4 * M * (M + 1) + 21 * M + 49)
    if kind == "adjoint":
        return {"bytes": 8.0 * n * N * (4 + 2 * case["steps"]), "flops": 5.0 * n * case["steps"] * attempt}
    if kind == "rkdp":
        return {"bytes": 16.0 * n * N * case["steps"], "flops": 2.0 * n * case["steps"] * (6 * rhs + 40 * N)}
    attempts = max(15.0, {"small": 75.0, "flame1d": 280.0, "batched": 43.0}[case["mech"]] * case["dt"] / 1e-6)
    if kind == "split":  # half the flame is cold
        attempts = 15.0
    return {"bytes": 16.0 * n * N * case["steps"], "flops": n * case["steps"] * attempts * attempt}


# ---------------------------------------------------------------- the same in plain float64 torch
R_GAS = 8.314462618
GAM = 0.572816062482135
G = ((), (-0.602765307997356,), (-1.389195789724843, 1.072950969011413),
     (0.992356412977094, -1.390032613873701, -0.440875890223325))
A = ((), (0.432364435748567,), (-0.514211316876170, 1.382271144617360))
B = (0.194335256262729, 0.483167813989227, 0.0, 0.322496929748044)
BH = (-0.217819895945721, 1.03130847478467, 0.186511421161047, 0.0)


class _Plain:
    """The source term of a mechanism on rows of cells, in float64."""

    def __init__(self, d, dev):
        t = lambda x: torch.as_tensor(np.asarray(x, dtype=np.float64), device=dev)  # noqa: E731
        self.ns, nr = d.n_species, d.n_reactions
        self.W, self.Tmid = t(d.W), t(d.nasa[:, 1])
        self.lo, self.hi = t(d.nasa[:, 3:10].T), t(d.nasa[:, 10:17].T)
        slots = np.full((nr, 4), self.ns)
        nu = np.zeros((nr, self.ns + 1))
        mol = np.zeros(nr)
        for j in range(nr):
            at = [0, 2]
            for i in range(4):
                k, c = int(d.rxn_sp[j, i]), int(d.rxn_nu[j, i])
                if k < 0:
                    continue
                nu[j, k] += c
                mol[j] += max(0, -c)
                for _ in range(abs(c)):
                    slots[j, at[i // 2]] = k
                    at[i // 2] += 1
        self.slots = torch.as_tensor(slots.T.copy(), device=dev)
        self.nu = t(nu[:, :self.ns])
        self.dnu = self.nu.sum(1)
        self.rev = t(d.reversible)
        self.third, self.troe = t(d.kind == 1), np.flatnonzero(d.kind == 2)
        self.lnA0 = t(np.log(d.arrh[:, 0]) + (mol + (d.kind == 1) - 1) * math.log(1e-6))
        self.lnA_in = t(np.log(d.arrh[:, 0]))
        self.lnA = self.lnA0
        self.b, self.Ea = t(d.arrh[:, 1]), t(d.arrh[:, 2] / R_GAS)
        self.eff = t(d.eff)
        self.pressure = bool((d.kind > 0).any())
        if len(self.troe):
            f = d.falloff[self.troe]
            self.k0 = t(np.log(f[:, 0]) + mol[self.troe] * math.log(1e-6)), t(f[:, 1]), t(f[:, 2] / R_GAS)
            self.fc = tuple(t(f[:, i]) for i in (3, 4, 5, 6))
            self.troe = torch.as_tensor(self.troe, device=dev)

    def __call__(self, u, rho=None, src=None):
        Y, T = u[:, :-1], u[:, -1:]
        a = torch.where((T < self.Tmid)[None], self.lo[:, None, :], self.hi[:, None, :])
        lnT = T.log()
        cp = a[0] + T * (a[1] + T * (a[2] + T * (a[3] + T * a[4])))
        h = a[0] + T * (a[1] / 2 + T * (a[2] / 3 + T * (a[3] / 4 + T * a[4] / 5))) + a[5] / T
        s = a[0] * lnT + T * (a[1] + T * (a[2] / 2 + T * (a[3] / 3 + T * a[4] / 4))) + a[6]
        N = Y / self.W
        shift = 0.0
        if rho is None:
            rho = P_ATM / (R_GAS * T * N.sum(1, keepdim=True))
        else:
            rho, shift = rho[:, None], 1.0
        C = torch.cat([rho * N, torch.ones_like(T)], 1)
        k = (self.lnA + self.b * lnT - self.Ea / T).exp()
        if self.pressure:
            M = C[:, :-1] @ self.eff.T
        if len(self.troe):
            j, (al, T3, T1, T2) = self.troe, self.fc
            Pr = (self.k0[0] + self.k0[1] * lnT - self.k0[2] / T).exp() * M[:, j] / k[:, j]
            Fc = (1 - al) * (-T / T3).exp() + al * (-T / T1).exp() + torch.where(T2 > 0, (-T2 / T).exp(), 0.0)
            lF = Fc.log10()
            x = Pr.log10() - 0.4 - 0.67 * lF
            f1 = x / (0.75 - 1.27 * lF - 0.14 * x)
            k = k.index_copy(1, j, k[:, j] * Pr / (1 + Pr) * ((lF / (1 + f1 * f1)) * math.log(10.0)).exp())
        Kc = (-(h - s) @ self.nu.T + self.dnu * (101325.0 / (R_GAS * T)).log()).exp()
        i = self.slots
        q = k * (C[:, i[0]] * C[:, i[1]] - self.rev / Kc * C[:, i[2]] * C[:, i[3]])
        if self.pressure:
            q = torch.where(self.third > 0, M * q, q)
        om = q @ self.nu
        cb = (N * (cp - shift)).sum(1, keepdim=True)
        f = torch.cat([self.W * om / rho, -T * ((h - shift) * om).sum(1, keepdim=True) / (rho * cb)], 1)
        return f if src is None else f + src


def _basis(f, u, fn, M):
    """Arnoldi's orthonormal basis [cells, M, N] of the Krylov space of J(u) and fn, and H."""
    n, H = u.shape[0], {}
    q = [fn / fn.norm(dim=1, keepdim=True)]
    for j in range(M):
        w = torch.func.jvp(f, (u,), (q[j],))[1]
        for _ in range(2):
            hs = [(x * w).sum(1) for x in q]
            for i, hij in enumerate(hs):
                w = w - hij[:, None] * q[i]
                H[i, j] = H[i, j] + hij if (i, j) in H else hij
        if j + 1 < M:
            H[j + 1, j] = w.norm(dim=1)
            q.append(w / H[j + 1, j][:, None])
    zero = torch.zeros(n, dtype=u.dtype, device=u.device)
    return torch.stack(q, 1), torch.stack([torch.stack([H.get((i, j), zero) for j in range(M)], 1) for i in range(M)], 1)


def _attempt(f, u, fn, Q, H, h):
    """ROK4E's solution and its embedded one after a step h [cells, 1]."""
    inv = torch.linalg.inv(torch.eye(H.shape[1], dtype=u.dtype, device=u.device) - (h * GAM)[:, :, None] * H)
    k, fi = [], fn
    for i in range(4):
        if i in (1, 2):
            fi = f(u + h * sum(a * x for a, x in zip(A[i], k)))
        g = sum(c / GAM * x for c, x in zip(G[i], k)) if i else torch.zeros_like(u)
        z = Q @ (fi + g)[:, :, None]
        k.append(fi + (Q.transpose(1, 2) @ (inv @ z - z))[:, :, 0])
    return u + h * sum(c * x for c, x in zip(B, k)), u + h * sum(c * x for c, x in zip(BH, k))


def _integrate(plain, U, dt, M, h, rho, src):
    """Every row over dt with its own steps; h is the carried step (0: dt), updated in place."""
    U = U.clone()
    act = torch.arange(U.shape[0], device=U.device)
    hh = torch.where(h > 0, h, dt)
    t, lg = torch.zeros_like(hh), torch.zeros_like(hh)
    fn = Q = H = None
    due = torch.ones_like(act, dtype=torch.bool)
    while act.numel():
        f_of = lambda rows: (lambda x: plain(x, None if rho is None else rho[rows], None if src is None else src[rows]))  # noqa: E731
        if due.any():
            a = _basis(f_of(act[due]), U[act[due]], f_of(act[due])(U[act[due]]), M)
            new = (f_of(act[due])(U[act[due]]), *a)
            if fn is None:
                fn, Q, H = new
            else:
                fn[due], Q[due], H[due] = new
        u = U[act]
        hh = torch.minimum(hh, dt - t)
        us, uh = _attempt(f_of(act), u, fn, Q, H, hh[:, None])
        err = ((uh - us) / (ATOL + RTOL * us.abs())).square().mean(1).sqrt()
        le = err.clamp(min=1e-10).log2()
        ok = err <= 1.0
        fac = (0.8 * torch.exp2(0.1 * lg - 0.175 * le)).clamp(0.2, 5.0)
        U[act[ok]] = us[ok]
        t = torch.where(ok, t + hh, t)
        hh = torch.where(err.isfinite(), hh * fac, hh * 0.2)
        lg = torch.where(ok, le, lg)
        h[act[ok]] = hh[ok]
        stay = dt - t > 1e-12 * dt
        act, hh, t, lg, fn, Q, H, due = act[stay], hh[stay], t[stay], lg[stay], fn[stay], Q[stay], H[stay], ok[stay]
    return U


DP = ((1 / 5,), (3 / 40, 9 / 40), (44 / 45, -56 / 15, 32 / 9),
      (19372 / 6561, -25360 / 2187, 64448 / 6561, -212 / 729),
      (9017 / 3168, -355 / 33, 46732 / 5247, 49 / 176, -5103 / 18656),
      (35 / 384, 0.0, 500 / 1113, 125 / 192, -2187 / 6784, 11 / 84))
DP_E = (71 / 57600, 0.0, -71 / 16695, 71 / 1920, -17253 / 339200, 22 / 525, -1 / 40)


def _explicit(plain, U, dt, h):
    """Dormand-Prince 5(4) with the elementary controller."""
    U = U.clone()
    act = torch.arange(U.shape[0], device=U.device)
    hh = torch.where(h > 0, h, dt)
    t = torch.zeros_like(hh)
    while act.numel():
        u = U[act]
        hh = torch.minimum(hh, dt - t)
        k = [plain(u)]
        for row in DP:
            us = u + hh[:, None] * sum(c * x for c, x in zip(row, k))
            k.append(plain(us))
        err = (hh[:, None] * sum(c * x for c, x in zip(DP_E, k)) / (ATOL + RTOL * us.abs())).square().mean(1).sqrt()
        ok = err <= 1.0
        U[act[ok]] = us[ok]
        t = torch.where(ok, t + hh, t)
        hh = torch.where(err.isfinite(), hh * (0.9 * err.clamp(min=1e-10) ** -0.2).clamp(0.2, 5.0), hh * 0.2)
        h[act[ok]] = hh[ok]
        stay = dt - t > 1e-12 * dt
        act, hh, t = act[stay], hh[stay], t[stay]
    return U


def _transport(X, dx):
    P = torch.cat([X[:1], X, X[-1:]])
    return D_DIFF * (P[:-2] - 2.0 * X + P[2:]) / dx**2


def exact(case, seed):
    U = _state(case, seed)
    plain = _Plain(_mechanism(case["mech"]), U.device)
    kind = case["kind"]
    if kind == "rhs":
        return torch.cat([plain(x) for x in U.split(16384)])
    if kind == "jvp":
        V = _direction(U, seed)
        return torch.cat([torch.func.jvp(plain, (x,), (v,))[1] for x, v in zip(U.split(16384), V.split(16384))])
    if kind == "adjoint":
        w, lnA = _cotangent(case, U), plain.lnA_in.clone().requires_grad_(True)
        plain.lnA = plain.lnA0 + (lnA - plain.lnA_in)
        ends, g_u0, g_lnA = [], [], torch.zeros_like(lnA)
        for x, wx in zip(U.split(256), w.split(256)):
            u0 = x.clone().requires_grad_(True)
            u = u0
            for _ in range(case["steps"]):
                fn = plain(u)
                u = _attempt(plain, u, fn, *_basis(plain, u, fn, case["M"]), torch.full_like(u[:, :1], case["h"]))[0]
            ga, gu = torch.autograd.grad((u * wx).sum(), (lnA, u0), retain_graph=True)
            ends.append(u.detach())
            g_u0.append(gu)
            g_lnA += ga
        return {"U": torch.cat(ends), "g_lnA": g_lnA.cpu(), "g_u0": torch.cat(g_u0)}
    h = torch.zeros_like(U[:, -1])
    rho = _rho(case, U) if case.get("volume") else None
    dx, dt = LENGTH / case["cells"], case["dt"]
    for _ in range(case["steps"]):
        if kind == "rkdp":
            U = _explicit(plain, U, dt, h)
        elif kind == "rok4e":
            U = _integrate(plain, U, dt, case["M"], h, rho, None)
        else:
            Tn = _transport(U, dx)
            X = _integrate(plain, U, dt, case["M"], h, None, Tn)
            k = 0.5 * dt
            V = X + k * (_transport(X, dx) - Tn)
            V = 0.75 * X + 0.25 * (V + k * (_transport(V, dx) - Tn))
            U = X / 3.0 + 2.0 / 3.0 * (V + k * (_transport(V, dx) - Tn))
    return U
