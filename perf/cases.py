"""What the performance of this package is measured on.

Each case is one call (or a pair of calls) of the public entry points in
paper_1110_4903_gb300.chem, at a size and with options that its users run:

  step         Chem.advance: one implicit chemistry step of a field
  step-graph   the same, captured once with Chem.graph and launched
  step-host    Chem.advance_host on pinned host buffers
  step-segs    Chem.advance_segmented: the step in several launches
  fields       Chem.state_from_tpy, then Chem.temperature of the result
  solve        batched_solve: batched dense elimination

The step updates its state in place, so a pass first restores the state from
a copy, as the benchmark does.  The request server is not timed here: a
request runs in the step kernel's own code, and what a server adds (arrival
order, polling and linger times) is not a pass of fixed work.

`exact` computes the same results in FP64 with plain torch operations: the
mechanism arrays are the only thing it shares with the library.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_1110_4903_gb300 import chem, synth

R = 8.314462618        # J/(mol K)
PA = 101325.0          # Pa
TREF = 298.15          # K, reference of the formation energies
T_LO, T_HI = 200.0, 6000.0

METHODS = {"global": chem.LU_GLOBAL, "global_fma": chem.LU_GLOBAL_FMA, "onchip": chem.LU_ONCHIP}

# Mean Newton iterations of a cell, for the operation counts (36 and 64
# species: uniform fields at 1e-6 s; the front field is mostly cold gas).
MEAN_ITERS = {("uniform", 9): 5.0, ("uniform", 36): 44.0, ("uniform", 64): 60.0, ("front", 36): 4.0}


def listed():
    return [
        # one backward-Euler step of 1,024 cells, no substeps: the smallest
        # block that a solver hands over, where latency counts
        dict(name="h2-1k-onestep-fp64", op="step", species=9, cells=1024, dt=1e-7, mixed=False,
             substeps=False, field="uniform"),
        # the 9-species detonation field on a million cells, adaptive, FP64
        dict(name="h2-1M-fp64", op="step", species=9, cells=1 << 20, dt=1e-6, mixed=False,
             substeps=True, field="uniform"),
        # a ragged medium request of a simulation with long fluid steps
        dict(name="h2-20k-long-mixed", op="step", species=9, cells=20011, dt=1e-5, mixed=True,
             substeps=True, field="uniform"),
        # the headline: 36 species, 308 reactions, 2^18 cells, mixed precision
        dict(name="hc36-256k-mixed", op="step", species=36, cells=1 << 18, dt=1e-6, mixed=True,
             substeps=True, field="uniform"),
        # the same mechanism in plain FP64, a block of a decomposed domain
        dict(name="hc36-16k-fp64", op="step", species=36, cells=16387, dt=1e-6, mixed=False,
             substeps=True, field="uniform"),
        # the smallest request of the serving stream: 1,024 cells of 36 species
        dict(name="hc36-1k-mixed", op="step", species=36, cells=1024, dt=1e-6, mixed=True,
             substeps=True, field="uniform"),
        # uneven work: a hot band through cold gas, replayed as a CUDA graph
        dict(name="hc36-front-graph", op="step-graph", species=36, cells=1024 * 512, nx=1024, dt=1e-6,
             mixed=True, substeps=True, field="front"),
        # domain segmentation (Sec. 5.2 of the paper): 128 x 128 in 4 launches
        dict(name="hc36-front-segs", op="step-segs", species=36, cells=128 * 128, nx=128, segments=4,
             dt=1e-6, mixed=True, substeps=True, field="front"),
        # a host flow solver: state in pinned host memory, copied both ways
        dict(name="h2-256k-host-mixed", op="step-host", species=9, cells=1 << 18, dt=1e-6, mixed=True,
             substeps=True, field="uniform"),
        # initial condition of a field, and its temperature for output
        dict(name="hc36-512k-fields", op="fields", species=36, cells=(1 << 19) + 77),
        # the kinetics-only experiment of Sec. 5.2: many small systems in the
        # interleaved layout, scalar rounding order
        dict(name="solve-37-global", op="solve", method="global", n=37, systems=45653),
        # and fewer, larger systems in the contiguous layout
        dict(name="solve-100-onchip", op="solve", method="onchip", n=100, systems=6250),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step"] * 6 + ["fields"] + ["solve"] * 3)
    if kind == "fields":
        return dict(op="fields", species=rng.choice([9, 36, 64]), cells=_log(rng, 1000, 1 << 20))
    if kind == "solve":
        method = rng.choice(sorted(METHODS))
        n = _log(rng, 4, 160 if method == "onchip" else 200)
        most = min(1 << 20, int(8e8 / (8 * n * n)))
        return dict(op="solve", method=method, n=n, systems=_log(rng, 32, most))
    species = rng.choice([9, 9, 9, 36, 36, 36, 64])
    mixed = rng.random() < 0.6
    if species == 36 and rng.random() < 0.3:
        nx = rng.choice([64, 128, 200, 256])
        ny = _log(rng, 16, 512)
        op = rng.choice(["step", "step-graph", "step-segs"])
        c = dict(op=op, species=36, cells=nx * ny, nx=nx, dt=1e-6, mixed=mixed, substeps=True, field="front")
        if op == "step-segs":
            c["segments"] = rng.choice([2, 3, 4, 8])
        return c
    most = {9: 1 << 20, 36: 1 << 16, 64: 1 << 12}[species] // (1 if mixed else 4)
    op = rng.choice(["step", "step", "step-graph", "step-host"])
    dt = 10.0 ** rng.uniform(-8, -5 if species == 9 else -6)
    return dict(op=op, species=species, cells=_log(rng, 50, most), dt=dt, mixed=mixed, substeps=True,
                field="uniform")


# ---------------------------------------------------------------- inputs
@functools.lru_cache(None)
def _mech(species):
    if species == 9:
        return synth.h2_air_9sp()
    if species == 36:
        return synth.hydrocarbon_36sp()
    return synth.hydrocarbon_mechanism(64, 60, 20, 400, 64480, "hc-64sp-480r")


def _dev():
    return torch.device("cuda")


class _Thermo:
    """NASA-7 thermodynamics of a mechanism (plain torch, FP64)."""

    def __init__(self, m, dev):
        def t(a):
            return torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device=dev)
        self.M, self.tmid, self.a = t(m.molar_mass), t(m.t_range[:, 1]), t(m.nasa7)
        self.ef = self.energies(torch.full((1,), TREF, dtype=torch.float64, device=dev))[0]

    def cpR_hRT_sR(self, T):
        T = T[:, None]
        a = torch.where((T > self.tmid)[:, :, None], self.a[:, 1], self.a[:, 0])
        a0, a1, a2, a3, a4, a5, a6 = a.unbind(2)
        cp = a0 + T * (a1 + T * (a2 + T * (a3 + T * a4)))
        h = a0 + T * (a1 / 2 + T * (a2 / 3 + T * (a3 / 4 + T * a4 / 5))) + a5 / T
        s = a0 * torch.log(T) + T * (a1 + T * (a2 / 2 + T * (a3 / 3 + T * a4 / 4))) + a6
        return cp, h, s

    def energies(self, T):
        """Energy per unit mass with its formation part, [cells, species]."""
        return R / self.M * T[:, None] * (self.cpR_hRT_sR(T)[1] - 1.0)

    def state(self, T, P, Y):
        """rho [species, cells], e [cells] of temperature, pressure and mass fractions."""
        rho = torch.empty_like(Y)
        e = torch.empty_like(T)
        for i in range(0, T.numel(), 1 << 16):
            j = slice(i, i + (1 << 16))
            y = Y[:, j].T
            r = (P[j] / (R * T[j] * (y / self.M).sum(1)))[:, None] * y
            rho[:, j] = r.T
            e[j] = (r * (self.energies(T[j]) - self.ef)).sum(1)
        return rho, e

    def temperature(self, rho, e, guess):
        """(T, ok) of [cells, species] densities and energies: Newton
        safeguarded by bisection on [T_LO, T_HI]."""
        T = torch.where((guess > T_LO) & (guess < T_HI), guess, torch.full_like(guess, 1500.0))
        lo, hi = torch.full_like(T, T_LO), torch.full_like(T, T_HI)
        done = torch.zeros_like(T, dtype=torch.bool)
        ok = torch.zeros_like(done)
        for _ in range(50):
            cp, h, _ = self.cpR_hRT_sR(T)
            f = (rho * (R / self.M * T[:, None] * (h - 1.0) - self.ef)).sum(1) - e
            fp = (rho * (R / self.M * (cp - 1.0))).sum(1)
            zero = (f == 0) & ~done
            ok |= zero
            done |= zero
            hi = torch.where(~done & (f > 0), T, hi)
            lo = torch.where(~done & ~(f > 0), T, lo)
            Tn = T - f / fp
            Tn = torch.where((Tn > lo) & (Tn < hi), Tn, 0.5 * (lo + hi))
            near = (Tn - T).abs() <= 1e-13 * Tn
            T = torch.where(done, T, Tn)
            fin = ~done & near
            ok |= fin & (T > T_LO * (1 + 1e-9)) & (T < T_HI * (1 - 1e-9))
            done |= fin
            if bool(done.all()):
                break
        return T, ok


def _field(case, seed):
    """(T, P, Y) on the GPU: uniform T and Dirichlet(1) mass fractions, or a
    2-D field with a hot band."""
    dev = _dev()
    m = _mech(case["species"])
    n = case["cells"]
    if case.get("field") == "front":
        f = synth.front_field(m, nx=case["nx"], ny=n // case["nx"], seed=seed, band=max(4, case["nx"] // 32))
        return tuple(torch.tensor(a, device=dev) for a in (f.T, f.P, f.Y))
    g = torch.Generator(device=dev).manual_seed(seed)
    lo, hi = (1000.0, 2500.0) if case.get("substeps") is False else (900.0, 2800.0)
    T = lo + (hi - lo) * torch.rand(n, generator=g, device=dev, dtype=torch.float64)
    Y = -torch.log1p(-torch.rand((m.ns, n), generator=g, device=dev, dtype=torch.float64))
    Y /= Y.sum(0)
    return T, torch.full_like(T, 101325.0), Y


def _system(case, seed):
    """Random systems with a diagonal shift of 0.5 sqrt(n), [n_sys, n, n] and
    [n_sys, n]; interleaved (systems fastest) for the global methods."""
    dev = _dev()
    n, k = case["n"], case["systems"]
    g = torch.Generator(device=dev).manual_seed(seed)
    eye = 0.5 * n ** 0.5 * torch.eye(n, dtype=torch.float64, device=dev)
    if case["method"] == "onchip":
        A = torch.randn((k, n, n), generator=g, dtype=torch.float64, device=dev)
        A += eye
        return A, torch.randn((k, n), generator=g, dtype=torch.float64, device=dev)
    A = torch.randn((n, n, k), generator=g, dtype=torch.float64, device=dev)
    A += eye[:, :, None]
    return A, torch.randn((n, k), generator=g, dtype=torch.float64, device=dev)


class _State:
    pass


def prepare(case, seed):
    s = _State()
    s.case, s.op = case, case["op"]
    dev = _dev()
    if s.op == "solve":
        s.method = METHODS[case["method"]]
        s.A0, s.b0 = _system(case, seed)
        s.A, s.b = torch.empty_like(s.A0), torch.empty_like(s.b0)
        s.piv = torch.empty((case["systems"], case["n"]), dtype=torch.int32, device=dev)
        s.info = torch.empty(case["systems"], dtype=torch.int32, device=dev)
        return s
    m = _mech(case["species"])
    n = case["cells"]
    T, P, Y = _field(case, seed)
    if s.op == "fields":
        s.chem = chem.Chem(m)
        s.T, s.P, s.Y = T, P, Y
        s.rho, s.e, s.T_out = torch.empty_like(Y), torch.empty_like(T), torch.empty_like(T)
        return s
    # (one backward-Euler step: no halving allowed)
    s.chem = chem.Chem(m, precision=chem.MIXED if case["mixed"] else chem.FP64,
                       **({} if case["substeps"] else {"max_halvings": 0}))
    s.rho0, s.e0 = _Thermo(m, dev).state(T, P, Y)
    if s.op == "step-host":
        s.rho0, s.e0 = s.rho0.cpu(), s.e0.cpu()
        s.rho, s.e, s.T = (torch.empty(t.shape, dtype=torch.float64, pin_memory=True)
                           for t in (s.rho0, s.e0, s.e0))
        s.status = torch.empty(n, dtype=torch.int32, pin_memory=True)
        return s
    s.rho, s.e, s.T = torch.empty_like(s.rho0), torch.empty_like(s.e0), torch.empty_like(s.e0)
    s.status = torch.empty(n, dtype=torch.int32, device=dev)
    if s.op == "step-graph":
        s.graph = s.chem.graph(s.rho, s.e, case["dt"], T_out=s.T, status=s.status)
    return s


def run(s):
    c = s.case
    if s.op == "solve":
        s.A.copy_(s.A0)
        s.b.copy_(s.b0)
        chem.batched_solve(s.method, s.A, s.b, s.piv, s.info)
        return {"A": s.A, "b": s.b, "piv": s.piv, "info": s.info}
    if s.op == "fields":
        s.chem.state_from_tpy(s.T, s.P, s.Y, s.rho, s.e)
        s.chem.temperature(s.rho, s.e, s.T_out)
        return {"rho": s.rho, "e": s.e, "T": s.T_out}
    s.rho.copy_(s.rho0)
    s.e.copy_(s.e0)
    if s.op == "step-host":
        s.chem.advance_host(s.rho.numpy(), s.e.numpy(), c["dt"], T_out=s.T.numpy(), status=s.status.numpy())
    elif s.op == "step-graph":
        s.graph.launch()
    elif s.op == "step-segs":
        s.chem.advance_segmented(s.rho, s.e, c["dt"], -(-c["cells"] // c["segments"]), T_out=s.T,
                                 status=s.status)
    else:
        s.chem.advance(s.rho, s.e, c["dt"], T_out=s.T, status=s.status)
    return {"rho": s.rho, "e": s.e, "T": s.T, "status": s.status}


def work(case):
    """Bytes of the inputs and outputs, once each, and the floating-point
    operations (exponentials and divisions as one each)."""
    if case["op"] == "solve":
        n, k = case["n"], case["systems"]
        # the elimination and the two substitutions
        flops = sum((n - j - 1) * (1 + 2 * (n - j - 1)) for j in range(n)) + 2 * n * n
        return {"bytes": k * (16 * (n * n + n) + 4 * n + 4), "flops": float(flops) * k}
    m = _mech(case["species"])
    ns, nr, n = m.ns, m.nr, case["cells"]
    if case["op"] == "fields":
        # T, P, Y in, rho, e out; then rho, e in, T out.  Energies by a
        # polynomial of degree five; about four temperature iterations
        return {"bytes": n * 8 * (2 * ns + 3 + ns + 2), "flops": float(n) * ns * (18 + 4 * 22)}
    ntb = int((np.asarray(m.third_body) != 0).sum())
    unk = ns + 1
    per_iter = (25 * ns + 20 * nr + 2 * ns * ntb + 84 * nr + 12 * ns * ntb + 5 * unk * unk + 2 * unk * ns
                + 2 * unk ** 3 / 3 + 2 * unk * unk + 3 * unk + 2 * nr)
    iters = 4.0 if not case["substeps"] else MEAN_ITERS[case["field"], ns]
    return {"bytes": n * (16 * unk + 12), "flops": per_iter * iters * n}


# ------------------------------------------------------- exact results
class _Step:
    """The implicit chemistry step as its definition has it, batched over
    cells in plain torch FP64: backward Euler by Newton's method with the
    analytic Jacobian on all species and the energy, substeps halved on
    failure and doubled after success."""

    RTOL, ATOL, MAX_NEWTON, MAX_ATTEMPTS = 1e-10, 1e-12, 12, 1000

    def __init__(self, m, dev, kappa, max_halvings):
        self.th = _Thermo(m, dev)
        self.kappa, self.max_halvings = kappa, max_halvings
        ns, nr = m.ns, m.nr
        self.ns = ns
        fac = np.full((2, nr, 3), ns, np.int64)      # concentration factors, species ns is 1
        nu = np.zeros((2, nr, ns))
        for side, (sp, k) in enumerate(((m.reac_sp, m.reac_nu), (m.prod_sp, m.prod_nu))):
            for r in range(nr):
                q = 0
                for j in range(3):
                    if sp[r, j] >= 0:
                        nu[side, r, sp[r, j]] += k[r, j]
                        for _ in range(int(k[r, j])):
                            fac[side, r, q] = sp[r, j]
                            q += 1
        tb = np.asarray(m.third_body) != 0
        order = nu[0].sum(1) + tb

        def t(a, dtype=torch.float64):
            return torch.tensor(np.ascontiguousarray(a), dtype=dtype, device=dev)
        self.fac = t(fac, torch.int64)
        self.nu, self.dnu = t(nu[1] - nu[0]), t((nu[1] - nu[0]).sum(1))
        self.tb = t(tb, torch.bool)
        self.eff = t(np.where(tb[:, None], m.tb_eff, 0.0))
        self.lnA = torch.log(t(m.arr_A)) + (t(order) - 1.0) * math.log(1e-6)
        self.beta, self.EaR = t(m.arr_beta), t(m.arr_Ea) / R

    def source_and_jacobian(self, rho, T):
        """Sources [cells, n] and their Jacobian [cells, n, n], n = ns + 1."""
        th, ns = self.th, self.ns
        N = T.numel()
        cp, h, s = th.cpR_hRT_sR(T)
        Tc = T[:, None]
        c = rho / th.M
        c1 = torch.cat([c, torch.ones_like(c[:, :1])], 1)
        lnkf = self.lnA + self.beta * torch.log(Tc) - self.EaR / Tc
        lnKc = self.dnu * torch.log(PA / (R * Tc)) - (h - s) @ self.nu.T
        kf = torch.exp(lnkf)
        k = (kf, torch.exp(lnkf - lnKc))
        CM = torch.where(self.tb, c @ self.eff.T, torch.ones_like(kf))
        D = torch.zeros((N, kf.shape[1], ns + 1), dtype=torch.float64, device=T.device)   # dQ/dc
        rate = []
        for side, sign in ((0, 1.0), (1, -1.0)):
            f = [c1[:, self.fac[side, :, j]] for j in range(3)]
            rate.append(k[side] * f[0] * f[1] * f[2])
            for j in range(3):
                d = sign * CM * k[side] * f[(j + 1) % 3] * f[(j + 2) % 3]
                D.scatter_add_(2, self.fac[side, :, j][None, :, None].expand(N, -1, 1), d[:, :, None])
        q = rate[0] - rate[1]
        D = D[:, :, :ns]
        D += q[:, :, None] * self.eff
        dlnkf = self.beta / Tc + self.EaR / (Tc * Tc)
        dlnKc = (h @ self.nu.T - self.dnu) / Tc
        dQdT = CM * (rate[0] * dlnkf - rate[1] * (dlnkf - dlnKc))
        rhocv = (rho * (R / th.M * (cp - 1.0))).sum(1)
        esens = R / th.M * Tc * (h - 1.0) - th.ef
        dTdx = torch.cat([-esens / rhocv[:, None], 1.0 / rhocv[:, None]], 1)
        w = th.M * ((CM * q) @ self.nu)
        numass = (self.nu * th.M).T                                     # [ns, nr]
        J = torch.zeros((N, ns + 1, ns + 1), dtype=torch.float64, device=T.device)
        J[:, :ns, :ns] = torch.matmul(numass, D / th.M)
        J[:, :ns] += (dQdT @ numass.T)[:, :, None] * dTdx[:, None, :]
        J[:, ns] = -(th.ef[None, :, None] * J[:, :ns]).sum(1)
        return torch.cat([w, -(w @ th.ef)[:, None]], 1), J

    def advance(self, rho, e, dt):
        """rho [cells, ns], e [cells] -> rho, e, T after dt (a cell that fails
        keeps its state and input temperature)."""
        th, ns = self.th, self.ns
        n = e.numel()
        x0 = torch.cat([rho, e[:, None]], 1)
        x = x0.clone()
        tot = rho.sum(1)
        atol = (self.ATOL * tot)[:, None].repeat(1, ns + 1)
        atol[:, ns] = self.ATOL * (e.abs() + (rho * th.ef).abs().sum(1))
        T, ok = th.temperature(rho, e, torch.full_like(e, 1500.0))
        T_in = torch.where(ok, T, torch.full_like(T, math.nan))
        T0 = T.clone()
        x_end, T_end = x0.clone(), T_in.clone()
        alive = ok & (tot > 0) & torch.isfinite(x0).all(1)
        total = 1 << self.max_halvings
        zi = torch.zeros(n, dtype=torch.int64, device=e.device)
        level, t, attempts, k = zi.clone(), zi.clone(), zi.clone() + 1, zi.clone()
        prev = torch.full_like(e, math.inf)
        while True:
            i = alive.nonzero().flatten()
            if i.numel() == 0:
                break
            xi, xo, Ti, ki, li = x[i], x0[i], T[i], k[i], level[i]
            # (iterations after the first recover the iterate's temperature)
            Tr, okT = th.temperature(xi[:, :ns], xi[:, ns], Ti)
            bad = (ki > 0) & ~okT
            Ti = torch.where((ki > 0) & okT, Tr, Ti)
            h = dt * torch.pow(2.0, -li.double())
            w, J = self.source_and_jacobian(xi[:, :ns], Ti)
            A = torch.eye(ns + 1, dtype=torch.float64, device=e.device) - h[:, None, None] * J
            d, info = torch.linalg.solve_ex(A, -(xi - xo - h[:, None] * w))
            xn = xi + d
            bad |= (info != 0) | ~torch.isfinite(xn).all(1)
            norm = (d.abs() / (self.RTOL * xn.abs() + atol[i])).amax(1)
            norm = torch.where(torch.isfinite(norm), norm, torch.full_like(norm, math.inf))
            pv = prev[i]
            conv = norm <= 1.0
            if self.kappa > 0:
                conv |= (ki >= 1) & (norm < pv) & (norm * norm <= self.kappa * (pv - norm))
            conv &= ~bad
            bad |= ~conv & (((ki >= 2) & (norm >= pv)) | (ki + 1 >= self.MAX_NEWTON))
            Tc, okc = th.temperature(torch.where(conv[:, None], xn, xo)[:, :ns],
                                     torch.where(conv, xn[:, ns], xo[:, ns]), Ti)
            acc = conv & okc & ~(xn[:, :ns] < -atol[i][:, :ns]).any(1)
            bad |= conv & ~acc
            go = ~acc & ~bad
            # accepted: the substep's state; rejected: back to its start
            tn = t[i] + torch.where(acc, torch.full_like(li, total) >> li, torch.zeros_like(li))
            end = acc & (tn >= total)
            x_end[i[end]], T_end[i[end]] = xn[end], Tc[end]
            xo = torch.where(acc[:, None], xn, xo)
            To = torch.where(acc, Tc, T0[i])
            ln = torch.where(acc, (li - 1).clamp(min=0), torch.where(bad, li + 1, li))
            dead = end | (bad & (ln > self.max_halvings)) | (~go & (attempts[i] >= self.MAX_ATTEMPTS))
            ln = ln.clamp(max=self.max_halvings)
            for _ in range(self.max_halvings):
                ln = torch.where(~go & ((torch.full_like(ln, total) >> ln) > total - tn), ln + 1, ln)
                ln = ln.clamp(max=self.max_halvings)
            x0[i], T0[i], t[i], level[i] = xo, To, tn, ln
            x[i] = torch.where(go[:, None], xn, xo)
            T[i] = torch.where(go, Ti, To)
            k[i] = torch.where(go, ki + 1, torch.zeros_like(ki))
            prev[i] = torch.where(go, norm, torch.full_like(norm, math.inf))
            attempts[i] += (~go).long()
            alive[i[dead]] = False
        return x_end[:, :ns], x_end[:, ns], T_end


def exact(case, seed):
    dev = _dev()
    if case["op"] == "solve":
        A, b = _system(case, seed)
        if case["method"] != "onchip":
            A, b = A.permute(2, 0, 1).contiguous(), b.T.contiguous()
        lu = torch.empty_like(A)
        x = torch.empty_like(b)
        step = max(1, (1 << 24) // (case["n"] ** 2))
        for i in range(0, case["systems"], step):
            lu[i:i + step] = torch.linalg.lu_factor(A[i:i + step])[0]
            x[i:i + step] = torch.linalg.solve(A[i:i + step], b[i:i + step])
        if case["method"] != "onchip":
            lu, x = lu.permute(1, 2, 0), x.T
        return {"A": lu, "b": x, "piv": None, "info": None}
    m = _mech(case["species"])
    T, P, Y = _field(case, seed)
    th = _Thermo(m, dev)
    rho, e = th.state(T, P, Y)
    if case["op"] == "fields":
        return {"rho": rho, "e": e, "T": T}
    # (larger ones take longer than 20 seconds)
    if case["cells"] * m.ns > (2400000 if m.ns < 16 else 600000 if case["field"] == "front" else 220000):
        return None
    st = _Step(m, dev, 0.01 if case["mixed"] else 0.0, 20 if case["substeps"] else 0)
    step = max(64, (1 << 25) // (m.nr * m.ns))
    out = [st.advance(rho[:, i:i + step].T.contiguous(), e[i:i + step], case["dt"])
           for i in range(0, case["cells"], step)]
    r, ee, TT = (torch.cat([o[j] for o in out]) for j in range(3))
    out = {"rho": r.T, "e": ee, "T": TT, "status": None}
    return {k: v.cpu() if v is not None and case["op"] == "step-host" else v for k, v in out.items()}
