"""The performance cases of the framework: the calls a reacting-flow program makes, over
the sizes it makes them at.

Every case is one pass through the public binding (``chem.Context``) on inputs made from
the seeded recipes of ``chem_inputs``: the per-cell integrator in both precision variants
and both mechanism sizes, device and host buffers, ragged AMR batches, the Strang-split 1D
step, and the learned surrogate's inference and training.  The in-place entry points get a
fresh copy of the inputs on each pass, as a flow solver hands over a new state each step.

``exact`` restates the same algorithms in 64-bit torch without the package's code: the
right-hand side, the RK4(3)5[2R+]C step control, the MUSCL / HLL Euler step, the
surrogate's network and error test, and the training loop.
"""
from __future__ import annotations

import math
import os
import struct
import tempfile

import numpy as np
import torch

from chem_inputs import mechanism, workloads
from paper_2506_02602_gb300 import chem, roofline

DEV = "cuda"
RU, P_REF = 8.31446261815324, 101325.0
RTOL, ATOL = 1e-6, 1e-10
SLICE_DT = 2e-9          # the detonation slice's hydro step
GATE = {"ood_margin": 0.05, "resid_max": 0.02, "neg_tol": 1e-6, "max_dT": 200.0, "err_tol": 6e-4, "rate_max": 1.5}


def listed():
    return [
        # one small patch of a flow: 256 reactors, where launch and one cell's latency count
        {"name": "reactors_256_fp64", "kind": "reactors", "n": 256, "variant": "fp64", "dt": 1e-7},
        # the benchmark's independent reactors, less than one wave of the GPU
        {"name": "reactors_4096_fp64", "kind": "reactors", "n": 4096, "variant": "fp64", "dt": 1e-7},
        # the benchmark's detonation slice, all cells of one level in one call, in both variants
        {"name": "slice_1m_fp64", "kind": "slice", "nx": 1024, "ny": 1024, "variant": "fp64"},
        {"name": "slice_1m_mixed", "kind": "slice", "nx": 1024, "ny": 1024, "variant": "mixed"},
        # the same slice handed over in host buffers, the copies inside the call
        {"name": "host_1m_mixed", "kind": "host", "nx": 1024, "ny": 1024, "variant": "mixed"},
        # an odd-sized slice of the 13-species mechanism
        {"name": "slice13_odd_mixed", "kind": "slice13", "nx": 401, "ny": 379, "variant": "mixed"},
        # the benchmark's ragged AMR batch (3 levels of subcycling, heavy-tailed stiffness)
        {"name": "amr_256_mixed", "kind": "amr", "boxes": 256, "variant": "mixed"},
        # a smaller ragged batch in fp64
        {"name": "amr_24_fp64", "kind": "amr", "boxes": 24, "variant": "fp64"},
        # one CFL-limited Strang step of a 1D detonation tube
        {"name": "strang_2048_fp64", "kind": "strang", "n": 2048, "variant": "fp64"},
        # surrogate inference: mildly reactive cells (nearly all accepted), and a longer step
        # where many cells go to the integrator
        {"name": "infer_2m_1e-9", "kind": "infer", "n": 2097152, "dt": 1e-9},
        {"name": "infer_300007_1e-8", "kind": "infer", "n": 300007, "dt": 1e-8},
        # surrogate training: epochs of 4096-row batches over a quarter million pairs
        {"name": "train_262144", "kind": "train", "pairs": 262144, "batch": 4096, "epochs": 5},
    ]


def draw(rng):
    def logint(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["reactors", "slice", "slice", "host", "slice13", "amr", "strang", "infer", "train"])
    variant = rng.choice(["fp64", "mixed"])
    if kind == "reactors":
        return {"kind": kind, "n": logint(32, 32768), "variant": variant, "dt": math.exp(rng.uniform(math.log(1e-8), math.log(1e-7)))}
    if kind in ("slice", "host", "slice13"):
        n, nx = logint(4096, 1 << 20), rng.randint(61, 1031)
        return {"kind": kind, "nx": nx, "ny": max(1, n // nx), "variant": variant}
    if kind == "amr":
        return {"kind": kind, "boxes": rng.randint(5, 40), "variant": variant}
    if kind == "strang":
        return {"kind": kind, "n": logint(200, 16384), "variant": variant}
    if kind == "infer":
        return {"kind": kind, "n": logint(5000, 2000000), "dt": math.exp(rng.uniform(math.log(1e-9), math.log(1e-8)))}
    return {"kind": kind, "pairs": logint(16384, 262144), "batch": rng.choice([2048, 4096, 4096]), "epochs": rng.randint(2, 5)}


# ---- inputs ---------------------------------------------------------------------------

def _f64(a):
    return torch.as_tensor(np.ascontiguousarray(a, dtype=np.float64), device=DEV)


def _mech(case):
    return mechanism.build13(0) if case["kind"] == "slice13" else mechanism.build(0)


class _Thermo:
    """NASA-7 mixture thermodynamics and rate tables of a mechanism as 64-bit tensors."""

    def __init__(self, m):
        self.m = m
        lo, hi = _f64(m["nasa_lo"]), _f64(m["nasa_hi"])
        self.W, self.Tm = _f64(m["W"])[:, None], float(m["T_mid"][0])
        s = torch.tensor([1, 1 / 2, 1 / 3, 1 / 4, 1 / 5, 1.0], device=DEV, dtype=torch.float64)
        one = torch.tensor([1, 0, 0, 0, 0, 0], device=DEV, dtype=torch.float64)
        # e_k / R_u per unit mass, and g_k / (R_u T), as polynomial coefficients [2, 6/7, S]
        self.ec = torch.stack([((a[:, :6] - one) * s / self.W).T for a in (lo, hi)])
        g = torch.tensor([1, -1 / 2, -1 / 6, -1 / 12, -1 / 20, 1, -1], device=DEV, dtype=torch.float64)
        self.gc = torch.stack([(a * g).T for a in (lo, hi)])
        S, R = len(m["W"]), len(m["A"])
        self.net = _f64(m["nu_r"] - m["nu_f"])
        self.rev = _f64(m["reversible"])[:, None]
        self.dnu = self.net.sum(1, keepdim=True)

        def molecules(nu):
            idx = np.full((2, R), S)
            for j in range(R):
                mol = [k for k in range(S) for _ in range(int(nu[j, k]))]
                idx[:len(mol), j] = mol
            return torch.as_tensor(idx, device=DEV)
        self.f_idx, self.r_idx = molecules(m["nu_f"]), molecules(m["nu_r"])
        col = lambda a: _f64(a)[:, None]  # noqa: E731
        self.lnA, self.b, self.Ta = col(np.log(m["A"])), col(m["b"]), col(m["Ea"] / RU)
        self.tb = torch.as_tensor(np.flatnonzero(m["rtype"] == 1), device=DEV)
        self.fo = torch.as_tensor(np.flatnonzero(m["rtype"] == 2), device=DEV)
        fo = np.flatnonzero(m["rtype"] == 2)
        self.eff = _f64(m["eff"])
        self.lnA0, self.b0, self.Ta0 = col(np.log(m["A0"][fo])), col(m["b0"][fo]), col(m["Ea0"][fo] / RU)
        self.troe, self.troe4 = _f64(m["troe"][fo]), _f64(m["troe_n"][fo] == 4)[:, None]

    def state(self, T, p, Y):
        rho = p / (RU * T * (Y / self.W).sum(0))
        return rho, RU * self.e_over_R(self.mix(Y), T)

    def mix(self, Y):
        return torch.einsum("rcs,sn->rcn", self.ec, Y)

    def e_over_R(self, mix, T, cv=False):
        c = torch.where(T >= self.Tm, mix[1], mix[0])
        e = ((((c[4] * T + c[3]) * T + c[2]) * T + c[1]) * T + c[0]) * T + c[5]
        return (e, (((5 * c[4] * T + 4 * c[3]) * T + 3 * c[2]) * T + 2 * c[1]) * T + c[0]) if cv else e

    def solve_T(self, Y, eR, T):
        mix = self.mix(Y)
        T = torch.where(T > 0, T, 1500.0)
        for _ in range(12):
            e, cv = self.e_over_R(mix, T, cv=True)
            d = (e - eR) / cv
            T = T - d
            if not bool(((d.abs() > 1e-13 * T) & torch.isfinite(d)).any()):
                break
        return torch.where((T > 0) & torch.isfinite(T) & (d.abs() <= 1e-9 * T), T, float("nan"))

    def gibbs(self, T):
        c = torch.where(T >= self.Tm, self.gc[1][:, :, None], self.gc[0][:, :, None])
        return c[0] * (1 - T.log()) + (((c[4] * T + c[3]) * T + c[2]) * T + c[1]) * T + c[5] / T + c[6]

    def rates(self, Y, rho, T):
        """dY/dt at temperature T."""
        lnT, c = T.log(), (rho * Y / self.W).clamp(min=0)
        kf = torch.exp(self.lnA + self.b * lnT - self.Ta / T)
        M = self.eff @ c
        k0 = torch.exp(self.lnA0 + self.b0 * lnT - self.Ta0 / T)
        Pr = k0 * M[self.fo] / kf[self.fo]
        a, t3, t1, t2 = (self.troe[:, i:i + 1] for i in range(4))
        lF = torch.log10((1 - a) * torch.exp(-T / t3) + a * torch.exp(-T / t1) + self.troe4 * torch.exp(-t2 / T))
        x = torch.log10(Pr) - 0.4 - 0.67 * lF
        f1 = x / (0.75 - 1.27 * lF - 0.14 * x)
        k = kf[self.fo] * Pr / (1 + Pr) * 10 ** (lF / (1 + f1 * f1))
        kf[self.fo] = torch.where(Pr > 0, k, 0.0)
        kr = self.rev * kf * torch.exp(self.net @ self.gibbs(T) + self.dnu * torch.log(RU * T / P_REF))
        cx = torch.cat([c, torch.ones_like(c[:1])])
        q = kf * cx[self.f_idx[0]] * cx[self.f_idx[1]] - kr * cx[self.r_idx[0]] * cx[self.r_idx[1]]
        q[self.tb] *= M[self.tb]
        return self.W * (self.net.T @ q) / rho

    def integrate(self, rho, e, Y, T, dt, nsub=None, max_steps=100000):
        """The two-register RK4(3)5[2R+]C scheme with WRMS step control over nsub steps of dt per cell."""
        A = (970286171893 / 4311952581923, 6584761158862 / 12103376702013, 2251764453980 / 15575788980749,
             26877169314380 / 34165994151039, 0.0)
        B = (1153189308089 / 22510343858157, 1772645290293 / 4653164025191, -1672844663538 / 4480602732383,
             2114624349019 / 3568978502595, 5198255086312 / 14908931495163)
        Bh = (1016888040809 / 7410784769900, 11231460423587 / 58533540763752, -1563879915014 / 6823010717585,
              606302364029 / 971179775848, 1097981568119 / 3980877426909)
        Yo, To = Y.clone(), T.clone()
        n = T.numel()
        idx, eR = torch.arange(n, device=DEV), e / RU
        dt = torch.full_like(T, dt) if isinstance(dt, float) else dt
        left = torch.ones(n, dtype=torch.int64, device=DEV) if nsub is None else nsub.to(torch.int64)
        s = {"rho": rho, "eR": eR, "T": T.clone(), "h": dt.clone(), "t": torch.zeros_like(T), "dt": dt, "left": left}
        X = Y.clone()
        for it in range(max_steps):
            h = torch.minimum(s["h"], s["dt"] - s["t"])
            U, Xn, E, Tn, Tacc = X, X, torch.zeros_like(X), s["T"], None
            for i in range(5):
                Tn = self.solve_T(U, s["eR"], Tn)
                Tacc = Tn if Tacc is None else Tacc
                F = self.rates(U, s["rho"], Tn)
                E = E + h * (B[i] - Bh[i]) * F
                U, Xn = Xn + h * A[i] * F, Xn + h * B[i] * F
            err = (E / (RTOL * torch.maximum(X.abs(), Xn.abs()) + ATOL)).square().mean(0).sqrt()
            fac = torch.where(err == 0, 5.0, (0.9 * err ** -0.25).clamp(0.2, 5.0))
            fac = torch.where(torch.isfinite(err), fac, 0.2)
            ok = err <= 1
            X = torch.where(ok, Xn, X)
            s["T"] = torch.where(ok, Tn, Tacc)
            s["t"] = s["t"] + torch.where(ok, h, 0.0)
            s["h"] = h * fac
            end = s["dt"] - s["t"] <= 1e-12 * s["dt"]
            s["left"] = s["left"] - end.to(torch.int64)
            s["t"] = torch.where(end, 0.0, s["t"])
            live = s["left"] > 0
            if it % 4 == 0 or idx.numel() < 20000:
                k = int(live.sum())
                if k < idx.numel():
                    d = ~live
                    Yo[:, idx[d]], To[idx[d]] = X[:, d], s["T"][d]
                    idx, X, s = idx[live], X[:, live], {q: v[live] for q, v in s.items()}
                if k == 0:
                    break
            else:  # finished cells idle until the next compaction
                s["dt"] = torch.where(live, s["dt"], 1e-30)
                s["left"] = torch.where(live, s["left"], 0)
        return Yo, self.solve_T(Yo, eR, To)


_TABLES = {}


def _thermo(case):
    k = "13" if case["kind"] == "slice13" else "9"
    if k not in _TABLES:
        _TABLES[k] = _Thermo(_mech(case))
    return _TABLES[k]


def _cells(case, seed):
    """(rho, e, buffer of Y planes and T, recipe dict) of a cell workload."""
    k = case["kind"]
    if k == "reactors":
        d = workloads.reactors(case["n"], seed=seed)
    elif k == "slice13":
        d = workloads.detonation_slice13(case["nx"], case["ny"], seed=seed)
    elif k == "amr":
        d = workloads.amr_batch(case["boxes"], seed=2)  # the boxes' sizes stay; the field takes +-2 % seeded noise
        noise = 1 + 0.02 * np.random.default_rng(seed).uniform(-1, 1, (2, d["T"].size))
        d["T"], d["p"] = d["T"] * noise[0], d["p"] * noise[1]
    else:
        d = workloads.detonation_slice(case["nx"], case["ny"], seed=seed)
    T, Y = _f64(d["T"]), _f64(d["Y"])
    rho, e = _thermo(case).state(T, _f64(d["p"]), Y)
    return rho, e, torch.cat([Y, T[None]]).contiguous(), d


def _tube(case, seed):
    """A 1D detonation tube: the slice's profile along x, the shocked gas moving at 1500 m/s (+-2 %)."""
    n = case["n"]
    d = workloads.detonation_slice(n, 1, seed=seed)
    T, Y = _f64(d["T"]), _f64(d["Y"])
    rho, e = _thermo(case).state(T, _f64(d["p"]), Y)
    shocked = np.arange(n) >= int(round(0.25 * n))
    u = _f64(np.where(shocked, -1500.0, 0.0) * (1 + 0.02 * np.random.default_rng(seed).uniform(-1, 1, n)))
    return torch.cat([rho[None], (rho * u)[None], (rho * (e + 0.5 * u * u))[None], rho * Y, T[None]]).contiguous()


# cells of the surrogate's family: H2-air at 900 - 2200 K and 1 - 30 atm, half of them with
# H, O and OH seeds between 1e-9 and 1e-5 (mole), as along an induction zone
def _induction_cells(th, n, seed):
    g = torch.Generator(device=DEV).manual_seed(seed)
    u = lambda lo, hi: lo + (hi - lo) * torch.rand(n, generator=g, device=DEV, dtype=torch.float64)  # noqa: E731
    phi, T, p = u(0.5, 2.0), u(900.0, 2200.0), u(1.0, 30.0) * P_REF
    X = torch.zeros(9, n, device=DEV, dtype=torch.float64)
    X[0], X[1], X[8] = 2 * phi, 1.0, 3.76
    X = X / X.sum(0)
    rad = torch.where(u(0, 1) < 0.5, 10 ** u(-9.0, -5.0), 0.0)
    X[3], X[4], X[5] = rad, rad, rad
    m = X * th.W
    Y = (m / m.sum(0)).contiguous()
    rho, e = th.state(T, p, Y)
    return rho, e, Y, T


def _boxcox(Y, lam=0.1):
    return (Y.clamp(min=1e-30) ** lam - 1) / lam


def _features(th, rho, Y, T, dt, lam=0.1):
    p = rho * RU * T * (Y / th.W).sum(0)
    dt = dt if isinstance(dt, torch.Tensor) else torch.full_like(T, dt)
    return torch.cat([torch.stack([T, p.log(), dt.log10()]), _boxcox(Y, lam)]).T


_NET = {}


def _net(th):
    """The surrogate a program has loaded: seeded random hidden layers and an output layer fitted by
    ridge regression to steps of the integrator, laid out as chem_surrogate_save writes it."""
    if not _NET:
        rng = np.random.default_rng(11)
        rho, e, Y, T = _induction_cells(th, 8192, 12345)
        dt = _f64(np.exp(rng.uniform(math.log(1e-9), math.log(1e-8), 8192)))
        Y1, _ = th.integrate(rho, e, Y, T, dt)
        X = _features(th, rho, Y, T, dt).cpu().numpy()
        D = ((_boxcox(Y1) - _boxcox(Y)) * (1e-8 / dt)).T.cpu().numpy()
        pad = lambda a, v=0.0: np.concatenate([a, np.full(16 - a.size, v)]).astype(np.float32)  # noqa: E731
        fstat = (X.mean(0), 1 / np.maximum(X.std(0), 1e-6))
        tstat = (D.mean(0), 1 / np.maximum(D.std(0), 1e-6))
        bf = lambda a: torch.as_tensor(a, dtype=torch.float32).bfloat16().double().numpy()  # noqa: E731
        H, layers = bf((X - fstat[0]) * fstat[1]), []
        for k, (fan, width) in enumerate([(12, 256), (256, 256), (256, 256)]):
            w = bf(rng.standard_normal((256, fan)) * math.sqrt(2 / fan))
            b = bf(rng.standard_normal(256) * 0.1)
            layers.append((np.pad(w, ((0, 0), (0, 4))) if k == 0 else w, b))
            H = torch.nn.functional.gelu(torch.as_tensor(H @ w.T + b)).numpy()
        Hb = np.concatenate([H, np.ones((H.shape[0], 1))], axis=1)
        out = np.linalg.solve(Hb.T @ Hb + 1e-3 * np.eye(257), Hb.T @ ((D - tstat[0]) * tstat[1]))
        w3, b3 = np.zeros((16, 256)), np.zeros(16)
        w3[:9], b3[:9] = bf(out[:256].T), bf(out[256])
        layers.append((w3, b3))
        flat = np.concatenate([np.concatenate([w.ravel(), b]) for w, b in layers]).astype(np.float32)
        head = b"CHEMSUR2" + struct.pack("<qdd", flat.size, 0.1, 1.0)
        norm = [pad(fstat[0]), pad(fstat[1]), X.min(0).astype(np.float32), X.max(0).astype(np.float32),
                pad(tstat[0]), pad(tstat[1])]
        _NET.update(file=head + b"".join(a.tobytes() for a in norm) + flat.tobytes(), layers=layers, norm=norm)
    return _NET


def _pairs(case, seed):
    """Training pairs: cells of the surrogate's family advanced over their own dt, 1e-9 - 1e-8 s."""
    th = _thermo(case)
    n = case["pairs"]
    rho, e, Y, T = _induction_cells(th, n, seed)
    g = torch.Generator(device=DEV).manual_seed(seed + 1)
    dt = 1e-9 * 10 ** torch.rand(n, generator=g, device=DEV, dtype=torch.float64)
    Y1, _ = th.integrate(rho, e, Y, T, dt)
    return rho, e, Y, T, dt, Y1.contiguous()


def prepare(case, seed):
    k = case["kind"]
    s = {"case": case}
    if k == "train":
        s["ctx"], s["pairs"] = chem.Context(_mech(case), "mixed"), _pairs(case, seed)
        return s
    if k == "infer":
        th = _thermo(case)
        s["ctx"] = chem.Context(_mech(case), "mixed")
        with tempfile.TemporaryDirectory() as d:
            path = os.path.join(d, "net.bin")
            with open(path, "wb") as f:
                f.write(_net(th)["file"])
            s["ctx"].surrogate_load(path)
        s["rho"], s["e"], Y, T = _induction_cells(th, case["n"], seed)
        s["in"] = torch.cat([Y, T[None]]).contiguous()
    elif k == "strang":
        s["ctx"], s["in"] = chem.Context(_mech(case), case["variant"]), _tube(case, seed)
    else:
        s["ctx"] = chem.Context(_mech(case), case["variant"])
        s["rho"], s["e"], s["in"], d = _cells(case, seed)
        if k == "amr":
            s["boxes"] = (torch.as_tensor(d["box_offset"], device=DEV), _f64(d["box_dt"]),
                          torch.as_tensor(d["box_nsub"], dtype=torch.int32, device=DEV))
        if k == "host":
            pin = lambda t: t.cpu().pin_memory()  # noqa: E731
            s["rho"], s["e"], s["in"] = pin(s["rho"]).numpy(), pin(s["e"]).numpy(), s["in"].cpu()
            s["buf"] = torch.empty_like(s["in"]).pin_memory()
            s["status"] = torch.empty(s["rho"].size, dtype=torch.int32).pin_memory().numpy()
            return s
    s["buf"] = torch.empty_like(s["in"])
    s["status"] = torch.zeros(s["in"].shape[1], dtype=torch.int32, device=DEV)
    return s


def run(s):
    case, ctx = s["case"], s["ctx"]
    k = case["kind"]
    if k == "train":
        rho, e, Y0, T0, dt, Y1 = s["pairs"]
        loss = ctx.surrogate_train(rho, e, Y0, dt, Y1, T0=T0, epochs=case["epochs"], batch=case["batch"], lr=1e-3,
                                   seed=1, dt_power=1.0)
        return {"loss": loss, "params": ctx.surrogate_params()}
    buf, status = s["buf"], s["status"]
    buf.copy_(s["in"])
    Y, T = buf[:-1], buf[-1]
    if k == "strang":
        U = {"rho": buf[0], "rhou": buf[1], "rhoE": buf[2], "rhoY": buf[3:-1], "T": T}
        dt = 0.45 * 25e-6 / ctx.euler1d_max_speed(U)
        ctx.strang_step(U, 25e-6, dt, (1, 0), RTOL, ATOL, status=status)
        return {"U": buf[:-1], "T": T, "status": status}
    if k == "host":
        ctx.integrate_host(s["rho"], s["e"], Y.numpy(), T.numpy(), SLICE_DT, RTOL, ATOL, status=status)
    elif k == "amr":
        ctx.integrate_batched(s["rho"], s["e"], Y, T, *s["boxes"], RTOL, ATOL, status=status)
    elif k == "infer":
        ctx.surrogate_infer(s["rho"], s["e"], Y, T, case["dt"], RTOL, ATOL, status=status)
    else:
        ctx.integrate(s["rho"], s["e"], Y, T, case.get("dt", SLICE_DT), RTOL, ATOL, status=status)
    return {"Y": Y, "T": T, "status": status}


def work(case):
    """State in and out once; the algorithm's floating-point work (attempted steps per cell of each
    recipe as the 64-bit algorithm takes them, each credited by the mechanism's structure)."""
    k = case["kind"]
    m = _mech(case)
    S = len(m["W"])
    if k == "train":
        steps = case["pairs"] // case["batch"] * case["epochs"]
        return {"bytes": case["pairs"] * 8.0 * (2 * S + 4), "flops": steps * case["batch"] * 3 * 278528.0}
    n = case.get("n") or case.get("nx", 0) * case.get("ny", 0) or 13504 * case["boxes"]
    if k == "infer":
        return {"bytes": n * (8.0 * (2 * S + 4) + 4), "flops": n * 278528.0}
    attempts = {"reactors": 3.1, "amr": 13.0, "strang": 15.0}.get(k, 7.4)
    per = roofline.step_flops(m)
    return {"bytes": n * (8.0 * (2 * S + 4) + 4), "flops": n * (attempts * per + roofline.cell_flops(m))}


# ---- the same in 64 bits --------------------------------------------------------------

def exact(case, seed):
    th, k = _thermo(case), case["kind"]
    if k == "train":
        return _train64(th, case, seed)
    if k == "infer":
        return _infer64(th, case, seed)
    if k == "strang":
        return _strang64(th, case, seed)
    rho, e, buf, d = _cells(case, seed)
    dt, nsub = case.get("dt", SLICE_DT), None
    if k == "amr":
        count = torch.as_tensor(np.diff(d["box_offset"]), device=DEV)
        dt = torch.repeat_interleave(_f64(d["box_dt"]), count)
        nsub = torch.repeat_interleave(torch.as_tensor(d["box_nsub"], device=DEV), count)
    Y, T = th.integrate(rho, e, buf[:-1], buf[-1], dt, nsub)
    return {"Y": Y, "T": T, "status": None}


def _prim64(th, U, T):
    rho, u = U[0], U[1] / U[0]
    Y = U[3:] / rho
    T = th.solve_T(Y, (U[2] / rho - 0.5 * u * u) / RU, T)
    return torch.cat([rho[None], u[None], (rho * RU * T * (Y / th.W).sum(0))[None], Y]), T


def _sound64(th, W, T):
    _, cv = th.e_over_R(th.mix(W[3:]), T, cv=True)
    return ((cv + (W[3:] / th.W).sum(0)) / cv * W[2] / W[0]).sqrt()


def _flux64(th, W, T):
    """HLL fluxes at the n + 1 faces: minmod slopes, a wall on the left and an open end on the right."""
    wall = lambda a, s: torch.cat([(a[:, :2] * s).flip(1), a, a[:, -1:], a[:, -1:]], 1)  # noqa: E731
    s = torch.ones_like(W[:, :1])
    s[1] = -1.0
    G, Tg = wall(W, s), wall(T[None], torch.ones_like(T[:1])[None])[0]
    d = G[:, 1:] - G[:, :-1]
    a, b = d[:, :-1], d[:, 1:]
    slope = torch.where(a * b <= 0, 0.0, torch.where(a.abs() < b.abs(), a, b))
    L, R = G[:, 1:-2] + 0.5 * slope[:, :-1], G[:, 2:-1] - 0.5 * slope[:, 1:]
    temp = lambda w: w[2] / (w[0] * RU * (w[3:] / th.W).sum(0))  # noqa: E731
    good = (L[0] > 0) & (L[2] > 0) & (R[0] > 0) & (R[2] > 0)
    TL, TR = torch.where(good, temp(L), Tg[1:-2]), torch.where(good, temp(R), Tg[2:-1])
    L, R = torch.where(good, L, G[:, 1:-2]), torch.where(good, R, G[:, 2:-1])

    def state(w, t):
        E = w[0] * (RU * th.e_over_R(th.mix(w[3:]), t) + 0.5 * w[1] ** 2)
        U = torch.cat([w[:1], (w[0] * w[1])[None], E[None], w[0] * w[3:]])
        F = U * w[1]
        F[1] += w[2]
        F[2] += w[2] * w[1]
        return F, U
    (FL, UL), (FR, UR), cL, cR = state(L, TL), state(R, TR), _sound64(th, L, TL), _sound64(th, R, TR)
    SL, SR = torch.minimum(L[1] - cL, R[1] - cR), torch.maximum(L[1] + cL, R[1] + cR)
    mid = (SR * FL - SL * FR + SL * SR * (UR - UL)) / (SR - SL)
    return torch.where(SL >= 0, FL, torch.where(SR <= 0, FR, mid))


def _strang64(th, case, seed):
    buf = _tube(case, seed)
    U, T = buf[:-1].clone(), buf[-1].clone()
    W, T1 = _prim64(th, U, T)
    dt = 0.45 * 25e-6 / float((W[1].abs() + _sound64(th, W, T1)).max())

    def chemistry(U, T):
        u = U[1] / U[0]
        Y, T = th.integrate(U[0], U[2] / U[0] - 0.5 * u * u, U[3:] / U[0], T, 0.5 * dt)
        return torch.cat([U[:3], U[0] * Y]), T
    U, T = chemistry(U, T)
    c = dt / 25e-6
    W, T = _prim64(th, U, T)
    F = _flux64(th, W, T)
    U1 = U + c * (F[:, :-1] - F[:, 1:])
    W, T = _prim64(th, U1, T)
    F = _flux64(th, W, T)
    U = 0.5 * (U + U1 + c * (F[:, :-1] - F[:, 1:]))
    U, T = chemistry(U, _prim64(th, U, T)[1])
    return {"U": U, "T": T, "status": None}


def _infer64(th, case, seed):
    """The surrogate's pass: network, element projection, temperature, gate and error test; the
    integrator for the cells that fail it."""
    net, dt, lam = _net(th), case["dt"], 0.1
    fmean, fistd, fmin, fmax, tmean, tistd = (_f64(a) for a in net["norm"])
    rho, e, Y0, T0 = _induction_cells(th, case["n"], seed)
    X = _features(th, rho, Y0, T0, dt, lam)
    span = GATE["ood_margin"] * (fmax - fmin)
    bad = ((X < fmin - span) | (X > fmax + span)).any(1)
    H = (X - fmean[:12]) * fistd[:12]
    for i, (w, b) in enumerate(net["layers"]):
        H = H @ _f64(w)[:, :H.shape[1]].T + _f64(b)
        H = torch.nn.functional.gelu(H) if i < 3 else H
    d = ((H[:, :9] / tistd[:9] + tmean[:9]) * (dt / 1e-8)).T
    y = Y0.clamp(min=1e-30)
    r = lam * d / (1 + lam * _boxcox(Y0, lam))
    Y = Y0 + y * torch.where(r > -1, torch.expm1(torch.log1p(r.clamp(min=-1 + 1e-12)) / lam), -1.0)
    mass = np.array([mechanism.ATOMIC_MASS[el] for el in mechanism.ELEMENTS])
    E = (th.m["ncomp"] * mass).T
    E = _f64(E / E.sum(0))
    res, Z = E @ (Y - Y0), E @ Y0
    bad |= ~(res.square().sum(0) <= GATE["resid_max"] ** 2 * Z.square().sum(0))
    w = Y.clamp(min=1e-12)
    M = torch.einsum("ak,kn,bk->nab", E, w, E)
    Y = Y - w * (E.T @ torch.linalg.solve(M, res.T[..., None])[..., 0].T)
    bad |= ~(Y >= -GATE["neg_tol"]).all(0)
    eR = e / RU
    T1 = th.solve_T(Y, eR, T0)
    bad |= ~((T1 - T0).abs() <= GATE["max_dT"])
    F0, F1 = th.rates(Y0, rho, T0), th.rates(Y, rho, T1)
    Ym = 0.5 * (Y0 + Y) + 0.125 * dt * (F0 - F1)
    Fm = th.rates(Ym, rho, th.solve_T(Ym, eR, 0.5 * (T0 + T1)))
    ec = torch.where(T1 >= th.Tm, th.ec[1][:, :, None], th.ec[0][:, :, None])
    uk = ((((ec[4] * T1 + ec[3]) * T1 + ec[2]) * T1 + ec[1]) * T1 + ec[0]) * T1 + ec[5]
    _, cv = th.e_over_R(th.mix(Y), T1, cv=True)
    est = ((uk - eR).abs() * (Y - Y0 - dt / 6 * (F0 + 4 * Fm + F1)).abs()).sum(0) / cv
    rate = dt * torch.maximum(F0.abs() / (Y0.abs() + 1e-6), F1.abs() / (Y.abs() + 1e-6)).amax(0)
    bad |= ~(rate <= GATE["rate_max"]) | ~(est <= GATE["err_tol"] * T1 * (1 - rate / 2 + rate * rate / 12))
    i = bad.nonzero()[:, 0]
    Y[:, i], T1[i] = th.integrate(rho[i], e[i], Y0[:, i], T0[i], dt)
    return {"Y": Y, "T": T1, "status": None}


def _splitmix(state, n):
    """n outputs of splitmix64 from a state (its increments are constant, so they vectorise)."""
    with np.errstate(over="ignore"):
        z = np.uint64(state) + np.arange(1, n + 1, dtype=np.uint64) * np.uint64(0x9E3779B97F4A7C15)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        return z ^ (z >> np.uint64(31))


def _train64(th, case, seed):
    """Adam on the mean squared error of the z-scored increments, the seeded initial weights and
    shuffles of the call (seed 1), cosine learning rate 1e-3 to 5e-5."""
    rho, _, Y0, T0, dt, Y1 = _pairs(case, seed)
    X = _features(th, rho, Y0, T0, dt)
    D = ((_boxcox(Y1) - _boxcox(Y0)) * (1e-8 / dt)).T
    X, D = ((a - a.mean(0)) / a.std(0, correction=0).clamp(min=1e-6) for a in (X, D))
    X = torch.nn.functional.pad(X, (0, 4))
    P, at = [], 0
    u = (_splitmix(0x2545F4914F6CDD1D + 1, 2 * (256 * 12 + 2 * 65536 + 9 * 256)) >> np.uint64(11)).astype(np.float64) / 2.0 ** 53
    nrm = np.sqrt(-2 * np.log(u[0::2] + 1e-300)) * np.cos(6.283185307179586 * u[1::2])
    for fan, out, wd, n in ((12, 256, 16, 256), (256, 256, 256, 256), (256, 256, 256, 256), (256, 9, 256, 16)):
        W = np.zeros((n, wd))
        W[:out, :fan] = math.sqrt(2 / fan) * nrm[at:at + out * fan].reshape(out, fan)
        at += out * fan
        P += [_f64(W).requires_grad_(), torch.zeros(n, device=DEV, dtype=torch.float64, requires_grad=True)]
    m, v = [torch.zeros_like(p) for p in P], [torch.zeros_like(p) for p in P]
    n, B, nb = case["pairs"], case["batch"], case["pairs"] // case["batch"]
    total, step, state, losses = nb * case["epochs"], 0, 1 ^ 0x5BD1E995, []
    for _ in range(case["epochs"]):
        j = (_splitmix(state, n - 1) % np.arange(n, 1, -1, dtype=np.uint64)).tolist()
        with np.errstate(over="ignore"):
            state = int(np.uint64(state) + np.uint64(n - 1) * np.uint64(0x9E3779B97F4A7C15))
        perm = list(range(n))
        for q, i in zip(j, range(n - 1, 0, -1)):
            perm[i], perm[q] = perm[q], perm[i]
        perm, loss = torch.as_tensor(perm, device=DEV), 0.0
        for b in range(nb):
            r = perm[b * B:(b + 1) * B]
            H = X[r]
            for i in range(4):
                H = H @ P[2 * i].T + P[2 * i + 1]
                H = torch.nn.functional.gelu(H) if i < 3 else H
            f = (H[:, :9] - D[r]).square().mean()
            g = torch.autograd.grad(f, P)
            loss = loss + f.detach()
            lr = 5e-5 + 0.5 * (1e-3 - 5e-5) * (1 + math.cos(math.pi * step / max(total - 1, 1)))
            step += 1
            with torch.no_grad():
                for p, gi, mi, vi in zip(P, g, m, v):
                    mi.mul_(0.9).add_(gi, alpha=0.1)
                    vi.mul_(0.999).addcmul_(gi, gi, value=0.001)
                    p -= lr * (mi / (1 - 0.9 ** step)) / ((vi / (1 - 0.999 ** step)).sqrt() + 1e-8)
        losses.append(float(loss) / nb)
    return {"loss": np.array(losses), "params": torch.cat([p.detach().ravel() for p in P])}
