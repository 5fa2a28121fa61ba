"""The work that users of this framework have it do, as measurable cases.

A flow solver calls the library once per time step: source terms or Jacobians of a field
(chem_rates, chem_jacobian), the stiff integration of every cell over the flow step
(chem_integrate and its variants), or the integration with its gradients (autograd.integrate).
The mechanisms are the repository's three synthetic ones: 10 species / 30 reactions, 53 / 325 (the
size of GRI-3.0) and 100 / 700.  Cell fields are drawn from the seed with the distributions of the
repository's workloads: Dirichlet mixtures over a temperature range, a mixing layer between two
streams, and a field of igniting, cold and burnt cells.  Flow steps run from 1e-10 s (compressible
direct simulation) to 1e-5 s (large-eddy simulation).
"""
from __future__ import annotations

import functools
import math
import time

import numpy as np
import torch

from paper_2105_12070_gb300 import autograd, chem, synth

P_ATM = 101325.0
RTOL, ATOL = 1e-6, 1e-10


def listed():
    return [
        # a reduced mechanism's source terms on one small block: launch latency
        dict(name="rates10_block", op="rates", mech=10, cells=256, field="uniform", p_atm=1.0),
        # source terms of a whole 256 x 256 mixing-layer field (an explicit or split scheme's call)
        dict(name="rates53_field", op="rates", mech=53, cells=65536, field="shear", p_atm=40.0),
        # Jacobians for an implicit flow solver or a time-scale analysis, a ragged block of cells
        dict(name="jacobian53_block", op="jacobian", mech=53, cells=2003, field="uniform", p_atm=20.0),
        # the repository's small configuration: 256 cells of the 10-species mechanism over 1e-5 s
        dict(name="step10_small", op="integrate", mech=10, cells=256, field="uniform", p_atm=1.0, dt=1e-5,
             variant="plain", precision="fp64", solver="rosenbrock"),
        # a flow step of a host code with a reduced mechanism: pinned host arrays in and out
        dict(name="step10_host", op="integrate", mech=10, cells=16384, field="uniform", p_atm=1.0, dt=1e-7,
             variant="host", precision="fp64", solver="rosenbrock"),
        # one well-mixed reactor (ignition delay, parameter studies): a single cell, latency only
        dict(name="reactor53_single", op="integrate", mech=53, cells=1, field="uniform", p_atm=13.5, dt=1e-7,
             variant="plain", precision="fp64", solver="rosenbrock"),
        # the headline configuration's mechanism and field on a block of cells
        dict(name="step53_shear", op="integrate", mech=53, cells=1000, field="shear", p_atm=40.0, dt=1e-8,
             variant="plain", precision="fp64", solver="rosenbrock"),
        # the same with the paper's integrator over a large-eddy time step
        dict(name="step53_seulex", op="integrate", mech=53, cells=1217, field="shear", p_atm=40.0, dt=1e-5,
             variant="plain", precision="fp64", solver="seulex"),
        # low-precision factors as a user selects them, a pressure per cell
        dict(name="step53_pairs", op="integrate", mech=53, cells=608, field="uniform", p_atm=20.0, dt=1e-9,
             variant="varp", precision="pairs", solver="rosenbrock"),
        # uneven stiffness: igniting, cold and burnt cells of the largest mechanism, the work queue's case
        dict(name="step100_uneven", op="integrate", mech=100, cells=203, field="uneven", p_atm=60.0, dt=1e-9,
             variant="plain", precision="fp64", solver="rosenbrock"),
        # sensitivities: forward solve with checkpoints and the reverse sweep, through autograd
        dict(name="gradient53", op="gradient", mech=53, cells=101, field="uniform", p_atm=20.0, dt=1e-10),
        # the same on the reduced mechanism over a longer step
        dict(name="gradient10", op="gradient", mech=10, cells=256, field="uniform", p_atm=1.0, dt=1e-6),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _log(rng, lo, hi):
    return float("%.3g" % math.exp(rng.uniform(math.log(lo), math.log(hi))))


def draw(rng):
    kind = rng.choice(["rates", "jacobian", "step10", "step53", "step53", "step100", "gradient10", "gradient53"])
    p = _log(rng, 1.0, 60.0)
    if kind in ("rates", "jacobian"):
        mech = rng.choice([10, 53, 100])
        most = {"rates": {10: 262144, 53: 65536, 100: 16384}, "jacobian": {10: 65536, 53: 4096, 100: 1024}}[kind][mech]
        field = rng.choice(["uniform", "shear"]) if mech != 100 else rng.choice(["uniform", "uneven"])
        return dict(op=kind, mech=mech, cells=_log_int(rng, 1, most), field=field, p_atm=p)
    if kind == "step10":
        return dict(op="integrate", mech=10, cells=_log_int(rng, 1, 16384), field=rng.choice(["uniform", "shear"]),
                    p_atm=p, dt=_log(rng, 1e-9, 1e-6), variant=rng.choice(["plain", "host", "varp"]),
                    precision=rng.choice(["fp64", "fp64", "pairs"]), solver=rng.choice(["rosenbrock", "seulex"]))
    if kind == "step53":
        solver = rng.choice(["rosenbrock", "rosenbrock", "seulex"])
        precision = rng.choice(["fp64", "fp64", "pairs", "refined"]) if solver == "rosenbrock" else "fp64"
        return dict(op="integrate", mech=53, cells=_log_int(rng, 1, 700), field=rng.choice(["uniform", "shear"]),
                    p_atm=p, dt=_log(rng, 1e-10, 1e-7), variant=rng.choice(["plain", "host", "varp"]),
                    precision=precision, solver=solver)
    if kind == "step100":
        return dict(op="integrate", mech=100, cells=_log_int(rng, 10, 150), field="uneven", p_atm=p,
                    dt=_log(rng, 1e-11, 1e-9), variant="plain", precision="fp64", solver="rosenbrock")
    mech = 10 if kind == "gradient10" else 53
    return dict(op="gradient", mech=mech, cells=_log_int(rng, 1, 256 if mech == 10 else 96), field="uniform", p_atm=p,
                dt=_log(rng, 1e-9, 1e-6) if mech == 10 else _log(rng, 1e-12, 1e-10))


# ------------------------------------------------------------------------------------------
# inputs


@functools.lru_cache(maxsize=None)
def _mechanism(K):
    m = {10: synth.mechanism_small, 53: synth.mechanism_53, 100: synth.mechanism_100}[K]()
    return m, m.write_temp()


def _cells(case, seed):
    """T [n], Y [K, n] of the case's field and the per-cell pressures in Pa."""
    K, n, field = case["mech"], case["cells"], case["field"]
    rng = np.random.default_rng([seed, 7])
    if field == "uniform":
        T, Y = synth.cells_uniform(seed, K, n, (1000.0, 1800.0) if K == 10 else (1000.0, 1300.0))
    elif field == "shear":
        nx = min(n, 256 if n >= 4096 else 4)
        ny = -(-n // nx)
        T, Y, _ = synth.cells_shear_layer(seed, K, nx, ny, delta=max(ny / 32.0, 0.25))
        T, Y = T[:n].copy(), Y[:, :n].copy()
    else:
        T, Y, _ = synth.cells_uneven(seed, K, n)
    p = case["p_atm"] * P_ATM * rng.uniform(0.9, 1.1, n)
    return T, np.ascontiguousarray(Y), p


def _cotangents(case, seed):
    rng = np.random.default_rng([seed, 8])
    n, K = case["cells"], case["mech"]
    return rng.standard_normal(n) * 1e-3, rng.standard_normal((K, n))


def _opts(case):
    kw = dict(use_queue=1)
    if case["solver"] == "seulex":
        kw["solver"] = chem.CHEM_SOLVER_SEULEX
    elif case["precision"] == "pairs":
        kw.update(precision=chem.CHEM_PREC_MIXED_FF, refine_sweeps=0)
    elif case["precision"] == "refined":
        kw.update(precision=chem.CHEM_PREC_MIXED, refine_sweeps=2)
    return chem.default_opts(**kw)


def prepare(case, seed):
    synthetic, path = _mechanism(case["mech"])
    T, Y, p = _cells(case, seed)
    s = dict(case=case, mech=chem.chem_load_mechanism(path), p=case["p_atm"] * P_ATM)
    n, K = case["cells"], case["mech"]
    if case["op"] == "integrate" and case["variant"] == "host":
        pin = lambda a: torch.from_numpy(a).pin_memory()
        s["T0"], s["Y0"] = pin(T), pin(Y)
        s["T"], s["Y"] = pin(np.empty_like(T)), pin(np.empty_like(Y))
        s["status"] = pin(np.zeros(n, np.int32))
        s["opts"] = _opts(case)
        return s
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    s["T0"], s["Y0"] = dev(T), dev(Y)
    if case["op"] == "rates":
        s["out"] = torch.empty((K, n), dtype=torch.float64, device="cuda")
    elif case["op"] == "jacobian":
        s["out"] = torch.empty((n, K, K), dtype=torch.float64, device="cuda")
    elif case["op"] == "integrate":
        s["T"], s["Y"] = torch.empty_like(s["T0"]), torch.empty_like(s["Y0"])
        s["status"] = torch.zeros(n, dtype=torch.int32, device="cuda")
        s["opts"] = _opts(case)
        s["p_cells"] = dev(p)
    else:
        gT, gY = _cotangents(case, seed)
        s["gT"], s["gY"] = dev(gT), dev(gY)
        s["lnA"] = dev(np.log(synthetic.A)).requires_grad_(True)
        s["T0"].requires_grad_(True)
        s["Y0"].requires_grad_(True)
    return s


def run(s):
    case, mech = s["case"], s["mech"]
    if case["op"] == "rates":
        return chem.chem_rates(mech, s["p"], s["T0"], s["Y0"], s["out"])
    if case["op"] == "jacobian":
        return chem.chem_jacobian(mech, s["p"], s["T0"], s["Y0"], s["out"])
    if case["op"] == "gradient":
        T, Y, status = autograd.integrate(mech, s["p"], s["T0"], s["Y0"], s["lnA"], case["dt"], rtol=RTOL, atol=ATOL)
        g = torch.autograd.grad((T, Y), (s["T0"], s["Y0"], s["lnA"]), (s["gT"], s["gY"]))
        return dict(T=T.detach(), Y=Y.detach(), status=status, gT0=g[0], gY0=g[1], g_lnA=g[2])
    # the flow solver hands over its field and takes the advanced one back, in place
    s["T"].copy_(s["T0"])
    s["Y"].copy_(s["Y0"])
    kw = dict(rtol=RTOL, atol=ATOL, status=s["status"], opts=s["opts"])
    if case["variant"] == "varp":
        chem.chem_integrate_varp(mech, s["p_cells"], s["T"], s["Y"], case["dt"], **kw)
    else:
        chem.chem_integrate(mech, s["p"], s["T"], s["Y"], case["dt"], **kw)
    return dict(T=s["T"], Y=s["Y"], status=s["status"])


# ------------------------------------------------------------------------------------------
# what a pass cannot do without, and how far two correct implementations are apart


def _attempts(case):
    """Step attempts per cell that the default tolerances take from these cold starts (typical
    counts, by field and flow step)."""
    x = math.log10(case["dt"])
    if case["mech"] == 10:
        pts = [(-9, 35), (-8, 150), (-7, 340), (-6, 500), (-5, 660)]
    elif case["mech"] == 100:
        pts = [(-11, 150), (-10, 350), (-9, 670), (-8, 1560)]
    else:
        pts = [(-12, 150), (-10, 600), (-9, 850), (-8, 1120), (-7, 1450), (-6, 1750), (-5, 2090)]
    return float(np.interp(x, [a for a, _ in pts], [b for _, b in pts]))


def _rate_flops(m):
    pd = int((m.rtype >= synth.TYPE_THIRD_BODY).sum())
    fo = int((m.rtype >= synth.TYPE_LINDEMANN).sum())
    return m.R * (2 * 25 + 14) + pd * 2 * m.K + fo * 200 + m.K * 40 + 2 * int(np.sum(m.reac >= 0) + np.sum(m.prod >= 0))


def _jacobian_flops(m):
    pd = int((m.rtype >= synth.TYPE_THIRD_BODY).sum())
    return _rate_flops(m) + 40 * m.R + 2 * 14 * m.R + 8 * pd * m.K + 8 * m.K * m.K


def work(case):
    m, _ = _mechanism(case["mech"])
    n, K = case["cells"], m.K
    state = 8 * n * (K + 1)
    if case["op"] == "rates":
        return dict(bytes=state + 8 * n * K, flops=n * _rate_flops(m))
    if case["op"] == "jacobian":
        return dict(bytes=state + 8 * n * K * K, flops=n * _jacobian_flops(m))
    lu, solve = 2.0 * K ** 3 / 3.0, 2.0 * K * K
    attempt = lu + 5 * solve + 2 * _rate_flops(m) + _jacobian_flops(m)
    steps = _attempts(case)
    if case["op"] == "gradient":
        back = lu + 8 * solve + 2 * _rate_flops(m) + 5 * _jacobian_flops(m)
        return dict(bytes=4 * state + 16 * m.R, flops=n * steps * (attempt + back))
    if case["solver"] == "seulex":
        # about a twelfth of the steps, each of about six columns
        return dict(bytes=2 * state, flops=n * max(steps / 12.0, 3.0) *
                    (_jacobian_flops(m) + 6 * lu + 21 * solve + 15 * _rate_flops(m)))
    return dict(bytes=2 * state, flops=n * steps * attempt)


def tolerance(case):
    # Measured between this library, an independent FP64 CPU implementation and runs with the inputs
    # and rate constants changed in the last bit.  Source terms and Jacobians differ by up to 1.5e-14.
    # The Rosenbrock solve repeats the same smooth sequence of step sizes: 4e-14 (largest value 1e-11)
    # on these cells, gradients 6e-13; an accepted step that turns into a rejected one, which a last-bit
    # change can bring on in a rare cell, costs a few times 1e-12 of a field.  Factors in FP32 pairs or FP32
    # carry 48 or 24 bits.  Seulex chooses its order and step by comparisons that a last-bit change
    # does turn over: 5.6e-8 (largest value 2e-6), inside its tolerance of 1e-6 per step.
    if case["op"] in ("rates", "jacobian"):
        return dict(rel=1e-13)
    if case["op"] == "gradient":
        return dict(rel=1e-11, max=1e-8)
    if case["solver"] == "seulex":
        return dict(rel=2.5e-7, max=1e-5)
    if case["precision"] != "fp64":
        return dict(rel=1e-9, max=1e-7)
    return dict(rel=1e-11, max=1e-9)


# ------------------------------------------------------------------------------------------
# the same quantities in plain torch, 64 bits


class _Plain:
    """Source term and Jacobian of a mechanism for a batch of cells, from its defining formulas."""

    RU, PATM = 8.314462618e7, 1.01325e6
    RC = 8.314462618 / 4.184  # cal/(mol K)

    def __init__(self, m, device):
        t = lambda a: torch.as_tensor(np.asarray(a, dtype=np.float64), device=device)
        self.K, self.R, self.dev = m.K, m.R, device
        self.W = t(m.W)
        self.lo, self.hi = t(m.a_low), t(m.a_high)
        nu = np.zeros((m.R, m.K))
        for side, sign in ((m.reac, -1.0), (m.prod, 1.0)):
            for u in range(2):
                ok = side[:, u] >= 0
                np.add.at(nu, (np.nonzero(ok)[0], side[ok, u]), sign)
        self.nu, self.dnu = t(nu), t(nu.sum(1))
        idx = lambda a: torch.as_tensor(np.where(a >= 0, a, m.K), device=device, dtype=torch.int64)  # K: the empty slot
        self.reac, self.prod = idx(m.reac), idx(m.prod)
        self.lnA, self.b, self.E = t(np.log(m.A)), t(m.b), t(m.Ea / self.RC)
        eff = np.zeros((m.R, m.K))
        low = np.zeros((m.R, 3))
        low[:, 0] = 1.0
        troe = np.tile([1.0, 1e30, 1e30, 1e30], (m.R, 1))
        for r in range(m.R):
            if m.rtype[r] >= synth.TYPE_THIRD_BODY:
                eff[r] = m.eff[r]
            if m.rtype[r] >= synth.TYPE_LINDEMANN:
                low[r] = m.low[r]
            if m.rtype[r] == synth.TYPE_TROE:
                troe[r] = m.troe[r]
        self.eff = t(eff)
        self.lnA0, self.b0, self.E0 = t(np.log(low[:, 0])), t(low[:, 1]), t(low[:, 2] / self.RC)
        self.troe = t(troe)
        kind = torch.as_tensor(m.rtype, device=device)
        self.third, self.fall = kind == synth.TYPE_THIRD_BODY, kind >= synth.TYPE_LINDEMANN
        self.is_troe = kind == synth.TYPE_TROE

    def thermo(self, T):
        T = T[:, None]
        a = torch.where((T <= synth.T_MID)[..., None], self.lo, self.hi)
        cp = a[..., 0] + T * (a[..., 1] + T * (a[..., 2] + T * (a[..., 3] + T * a[..., 4])))
        h = (a[..., 0] + T * (a[..., 1] / 2 + T * (a[..., 2] / 3 + T * (a[..., 3] / 4 + T * a[..., 4] / 5)))
             + a[..., 5] / T)
        s = (a[..., 0] * torch.log(T) + T * (a[..., 1] + T * (a[..., 2] / 2 + T * (a[..., 3] / 3 + T * a[..., 4] / 4)))
             + a[..., 6])
        dcp = a[..., 1] + T * (2 * a[..., 2] + T * (3 * a[..., 3] + T * 4 * a[..., 4]))
        return cp, h, s, dcp

    def constants(self, T, M):
        """Forward and reverse rate constants [n, R], with [M] of the plain third bodies included."""
        _, h, s, _ = self.thermo(T)
        T = T[:, None]
        lnT = torch.log(T)
        k = torch.exp(self.lnA + self.b * lnT - self.E / T)
        k0 = torch.exp(self.lnA0 + self.b0 * lnT - self.E0 / T)
        Pr = torch.where(self.fall, k0 * M / k, torch.ones_like(k))
        a, T3, T1, T2 = self.troe.unbind(1)
        Fc = (1 - a) * torch.exp(-T / T3) + a * torch.exp(-T / T1) + torch.exp(-T2 / T)
        L = torch.where(self.is_troe, torch.log10(torch.where(self.is_troe, Fc, torch.ones_like(Fc))), torch.zeros_like(Fc))
        x = torch.log10(Pr) - 0.4 - 0.67 * L
        f1 = x / (0.75 - 1.27 * L - 0.14 * x)
        F = torch.exp(math.log(10.0) * L / (1 + f1 * f1))
        kf = torch.where(self.fall, k * (Pr / (1 + Pr)) * F, torch.where(self.third, k * M, k))
        lnKc = -((h - s) @ self.nu.T) + self.dnu * torch.log(self.PATM / (self.RU * T))
        return kf, kf * torch.exp(-lnKc)

    def evaluate(self, p, phi, jacobian):
        """f [n, N] (and J [n, N, N]) at phi = [T, Y_1 .. Y_{K-1}]; p in Pa, per cell."""
        K, RU = self.K, self.RU
        T = phi[:, 0]
        Y = torch.cat([phi[:, 1:], 1 - phi[:, 1:].sum(1, keepdim=True)], 1)
        Wm = 1 / (Y / self.W).sum(1)
        rho = 10 * p * Wm / (RU * T)
        C = rho[:, None] * Y / self.W
        cpR, hRT, _, dcpR = self.thermo(T)
        M = C @ self.eff.T
        M = torch.where(self.third | self.fall, M, torch.ones_like(M))
        C1 = torch.cat([C, torch.ones_like(C[:, :1])], 1)
        r, q = C1[:, self.reac], C1[:, self.prod]  # [n, R, 2]
        pf, pr = r[..., 0] * r[..., 1], q[..., 0] * q[..., 1]
        if jacobian:
            Tm = T[:, None].expand_as(M)
            (kf, kr), (kfM, krM) = torch.func.jvp(lambda m: self.constants(T, m), (M,), (torch.ones_like(M),))
            _, (kfT, krT) = torch.func.jvp(lambda t: self.constants(t, M), (T,), (torch.ones_like(T),))
        else:
            kf, kr = self.constants(T, M)
        rate = kf * pf - kr * pr
        om = rate @ self.nu
        cp = RU * (Y * cpR / self.W).sum(1)
        H = hRT * RU * T[:, None]
        fT = -(H * om).sum(1) / (rho * cp)
        f = torch.cat([fT[:, None], (self.W * om / rho[:, None])[:, :-1]], 1)
        if not jacobian:
            return f
        n, N = T.shape[0], K
        dq = (kfM * pf - krM * pr)[..., None] * self.eff  # d rate / dC [n, R, K]
        dq = torch.cat([dq, torch.zeros_like(dq[..., :1])], 2)
        for idx, c, k, sign in ((self.reac, r, kf, 1.0), (self.prod, q, kr, -1.0)):
            for u in range(2):
                dq.scatter_add_(2, idx[None, :, u:u + 1].expand(n, -1, 1), (sign * k * c[..., 1 - u])[..., None])
        dq = dq[..., :K]
        domC = torch.einsum("rk,nrj->nkj", self.nu, dq)
        domT = (kfT * pf - krT * pr) @ self.nu
        # C_j = rho Y_j / W_j, rho = p Wm / (Ru T), all K mass fractions independent
        dlnrho = -Wm[:, None] / self.W  # d ln rho / dY_i
        domC_C = torch.einsum("nkj,nj->nk", domC, C)
        domY = domC * (rho[:, None] / self.W)[:, None, :] + domC_C[:, :, None] * dlnrho[:, None, :]
        domTt = domT - domC_C / T[:, None]
        # f_Yk = W_k om_k / rho, f_T = -sum H om / (rho cp)
        J = torch.zeros((n, 1 + K, 1 + K), dtype=phi.dtype, device=phi.device)
        g = self.W * om / rho[:, None]
        J[:, 1:, 1:] = self.W[:, None] * domY / rho[:, None, None] - g[:, :, None] * dlnrho[:, None, :]
        J[:, 1:, 0] = self.W * domTt / rho[:, None] + g / T[:, None]
        HdomY = torch.einsum("nk,nki->ni", H, domY)
        dcpY = RU * cpR / self.W
        J[:, 0, 1:] = -HdomY / (rho * cp)[:, None] - fT[:, None] * (dlnrho + dcpY / cp[:, None])
        dcpT = RU * (Y * dcpR / self.W).sum(1)
        J[:, 0, 0] = (-(H * domTt).sum(1) - RU * (cpR * om).sum(1)) / (rho * cp) + fT / T - fT * dcpT / cp
        J = J[:, :N, :]  # fold Y_K = 1 - sum of the others into the columns
        return f, J[:, :, :N] - torch.cat([torch.zeros_like(J[:, :, :1]), J[:, :, N:].expand(-1, -1, N - 1)], 2)

    def solve(self, p, phi, dt, most_s):
        """phi(dt), converged well below the default tolerances: the linearly implicit Euler method
        extrapolated to order 10 (Hairer & Wanner IV.9), a step size per cell, the columns of the
        tableau side by side in the batch.  None if it takes longer than most_s seconds."""
        began = time.monotonic()
        kmax, N = 10, phi.shape[1]
        phi = phi.clone()
        t = torch.zeros_like(phi[:, 0])
        h = torch.full_like(t, 1e-4 * dt)
        eye = torch.eye(N, dtype=phi.dtype, device=phi.device)
        col = torch.arange(1, kmax + 1, dtype=phi.dtype, device=phi.device)
        while True:
            act = torch.nonzero(t < dt)[:, 0]
            if act.numel() == 0:
                return phi
            if time.monotonic() - began > most_s:
                return None
            y0, ta, pa = phi[act], t[act], p[act]
            ha = torch.minimum(h[act], dt - ta)
            f0, J = self.evaluate(pa, y0, True)
            lu, piv = torch.linalg.lu_factor(eye * (col[:, None] / ha)[..., None, None] - J)  # [column, cell, N, N]
            y = y0.expand(kmax, -1, -1).clone()
            for sub in range(kmax):  # sub-step sub of the columns that have it
                if sub == 0:
                    f = f0.expand(kmax, -1, -1)
                else:
                    f = self.evaluate(pa.repeat(kmax - sub), y[sub:].reshape(-1, N), False).reshape(kmax - sub, -1, N)
                y[sub:] += torch.linalg.lu_solve(lu[sub:], piv[sub:], f[..., None])[..., 0]
            row = [y[0]]
            for j in range(2, kmax + 1):
                prev, row = row, [y[j - 1]]
                for i in range(1, j):
                    row.append(row[i - 1] + (row[i - 1] - prev[i - 1]) / (j / (j - i) - 1.0))
            scale = 1e-13 + 1e-9 * torch.maximum(y0.abs(), row[-1].abs())
            err = ((row[-1] - row[-2]).abs() / scale).amax(1)
            err = torch.where(torch.isfinite(err), err, torch.full_like(err, 1e20))
            ok = err <= 1.0
            phi[act] = torch.where(ok[:, None], row[-1], y0)
            t[act] = torch.where(ok, torch.where(ha >= dt - ta, torch.full_like(ta, dt), ta + ha), ta)
            h[act] = ha * (0.8 * err.clamp(min=1e-30) ** (-1.0 / kmax)).clamp(0.1, 4.0)


def exact(case, seed):
    m, _ = _mechanism(case["mech"])
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    T, Y, p = _cells(case, seed)
    plain = _Plain(m, dev)
    phi = torch.as_tensor(np.concatenate([T[None], Y[:-1]]).T.copy(), device=dev)
    n, K = phi.shape[0], m.K
    pressures = torch.full((n,), case["p_atm"] * P_ATM, dtype=torch.float64, device=dev)
    if case["op"] == "rates":
        out = torch.empty((K, n), dtype=torch.float64, device=dev)
        for c in range(0, n, 4096):
            out[:, c:c + 4096] = plain.evaluate(pressures[c:c + 4096], phi[c:c + 4096], False).T
        return out
    if case["op"] == "jacobian":
        out = torch.empty((n, K, K), dtype=torch.float64, device=dev)
        for c in range(0, n, 256):
            out[c:c + 256] = plain.evaluate(pressures[c:c + 256], phi[c:c + 256], True)[1]
        return out
    if n > {10: 2048, 53: 128, 100: 0}[case["mech"]]:  # more than about 20 seconds
        return None
    if case.get("variant") == "varp":
        pressures = torch.as_tensor(p, device=dev)
    end = plain.solve(pressures, phi, case["dt"], 18.0)
    if end is None:
        return None
    out = dict(T=end[:, 0].contiguous(), Y=torch.cat([end[:, 1:], 1 - end[:, 1:].sum(1, keepdim=True)], 1).T.contiguous(),
               status=torch.zeros(n, dtype=torch.int32, device=dev))
    if case["op"] == "gradient":
        out.update(gT0=None, gY0=None, g_lnA=None)
    return out
