"""The work that users of this framework have it do, as cases that can be timed and compared.

A case is a run, a batch of runs, or a gradient of a run:
  * step:    one lattice: initial fields, `steps` fused steps, the macroscopic fields back;
  * batch:   many lattices advanced together (Batch), the same three stages;
  * adjoint: loss and parameter gradient of a run (lbm_adjoint_fl_loss).
The problems, their sizes and parameters are those of `paper_2603_22902_gb300.workloads` (the film, the single
and the compound drop, the Janus drop, the pools, the drop sweep), with noise on the initial velocity and
temperature drawn from the seed.

The fields of a run come back in the storage type of its policy's populations (float64 for FP64 and double words,
float32 for FP32, float16 / bfloat16 for 16-bit storage): more digits than that a run does not hold.  The liquid
fraction is returned as that of the phase-changing material, phi_pcm f_l: f_l alone is 0 or 1 by the sign of a
rounding-level tail where there is no such material (cold gas).
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2603_22902_gb300 import lbm as L
from paper_2603_22902_gb300 import workloads as W
from paper_2603_22902_gb300.grad import pcm_liquid_fraction

_DTYPE = {"fp64": torch.float64, "df64": torch.float64, "fp32": torch.float32, "fp16s": torch.float16,
          "bf16s": torch.bfloat16}
_FIELDS = ("phi", "T", "H", "pcm_fl", "ux", "uy", "p")


def listed():
    def step(name, problem, nx, ny, precision, steps):
        return dict(name=name, kind="step", problem=problem, nx=nx, ny=ny, precision=precision, steps=steps)

    return [
        # the film problem at its own size: the smallest lattice in use, a run is launches and latency
        step("film_16x256_fp64", "film", 16, 256, "fp64", 100),
        # the Janus drop at the paper's size (N = 3): a middling lattice, cut by its tiles on both axes
        step("janus_300x150_fp64", "janus", 300, 150, "fp64", 40),
        # the single droplet, the benchmark's workload, in the parity policy ...
        step("drop_512_fp64", "drop", 512, 512, "fp64", 20),
        # ... in double words, the fast FP64-class policy ...
        step("drop_512_df64", "drop", 512, 512, "df64", 40),
        # ... and in 16-bit storage, for long forward studies
        step("drop_512_fp16s", "drop", 512, 512, "fp16s", 100),
        # a droplet on a lattice of odd sides: no row is aligned, no tile fits, the 16-bit copies cannot be used
        step("drop_509x387_fp16s", "drop", 509, 387, "fp16s", 60),
        # the compound drop at its own size (N = 3), in single precision ...
        step("compound_1024_fp32", "compound", 1024, 1024, "fp32", 20),
        # ... and in 16-bit storage
        step("compound_1024_fp16s", "compound", 1024, 1024, "fp16s", 20),
        # the largest lattice the measurements report: far beyond the L2 cache
        step("drop_2048_fp16s", "drop", 2048, 2048, "fp16s", 20),
        # a part of the droplet sweep (uneven sides 128 .. 512), in the form its tuner picks
        dict(name="sweep_32_fp16s", kind="batch", problem="sweep", cases=32, mode="staged", precision="fp16s", steps=20),
        # a few small parity runs side by side (walls, outflow, periodic sides, odd sizes)
        dict(name="small_batch_fp64", kind="batch", problem="small", cases=5, mode="per_step", precision="fp64",
             steps=40),
        # the gradient of the impurity problem (N = 4), with checkpoints and recomputation
        dict(name="adjoint_256_fp64", kind="adjoint", problem="impurity", nx=256, ny=256, precision="fp64", steps=20,
             checkpoint=5),
    ]


def draw(rng):
    log_int = lambda a, b: int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))
    u = rng.random()
    if u < 0.14:
        # parameter studies of any number of runs, in the forms a plan can have
        prec = rng.choice(["fp16s", "fp32", "fp64", "df64"])
        return dict(kind="batch", problem=rng.choice(["sweep", "small"]), cases=rng.randint(2, 24),
                    mode=rng.choice(["staged", "per_step", "persistent"]), precision=prec, steps=rng.randint(4, 20),
                    pick=rng.randint(1, 10 ** 6))
    if u < 0.26:
        # gradients: pools of other sizes, any checkpoint distance
        n = log_int(64, 288)
        return dict(kind="adjoint", problem="impurity", nx=n, ny=n + rng.randint(-8, 8), precision="fp64",
                    steps=rng.randint(3, 16), checkpoint=rng.randint(1, 8))
    problem = rng.choice(["film", "drop", "drop", "compound", "janus", "pool", "impurity"])
    nx, ny = log_int(48, 1400), log_int(48, 1400)
    if problem == "film":
        nx = log_int(4, 96)
    if problem in ("compound", "pool", "impurity"):
        ny = nx = max(nx, 64)
    if rng.random() < 0.5 and problem not in ("pool", "impurity"):
        nx = max(8, nx // 8 * 8)
    if problem == "pool":
        nx = ny = min(nx, 900)
    if problem == "impurity":
        nx = ny = min(nx, 640)
    prec = rng.choice(["fp64", "df64", "fp32", "fp16s", "fp16s", "bf16s"])
    c = dict(kind="step", problem=problem, nx=nx, ny=ny, precision=prec, steps=1)
    per_step = work(dict(c, steps=2))["bytes"] - work(c)["bytes"]
    c["steps"] = int(min(60, max(3, 6e9 * rng.uniform(0.2, 1.0) / per_step)))
    return c


# ---- inputs -------------------------------------------------------------------------------------------

_N = {"film": 2, "drop": 2, "compound": 3, "janus": 3, "pool": 3, "impurity": 4}


def _problem(problem, nx, ny, seed):
    """A workloads.Case of the given problem and size; its parameters are the workload's own."""
    if problem == "film":
        return W.film(nx=nx, ny=ny, h0=ny / 2.0)
    if problem == "drop":
        return W.sessile_drop(n=nx, ny=ny, R=0.195 * min(nx, 2 * ny))
    if problem == "compound":
        return W.compound_drop(n=nx, ny=ny, R_core=0.078 * nx, R_shell=0.156 * nx, seed=seed)
    if problem == "janus":
        return W.janus_drop(nx=nx, ny=ny, R=0.2 * min(nx, 2 * ny), mobility=0.1)
    if problem == "pool":
        return W.lateral_pool(n=nx, T0=0.5)
    if problem == "impurity":
        return W.impurity_freeze(n=nx, ny=ny, n_disks=max(2, min(24, nx * ny // 12000)))
    raise ValueError(problem)


def _batch(case):
    if case["problem"] == "sweep":
        return W.batch_sweep(n_cases=case["cases"], seed=case.get("pick", 4))
    few = W.small_batch()
    return [few[k % len(few)] for k in range(case["cases"])]


def _inputs(c, seed):
    """Initial fields on the GPU: the problem's own, with noise on the velocity and, where the run starts away
    from the melting point, on the temperature."""
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    dev = lambda a: torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")
    noise = lambda a: (torch.rand((c.ny, c.nx), generator=g, device="cuda", dtype=torch.float64) * 2.0 - 1.0) * a
    warm = float(c.T.min()) > c.T_liq
    return (dev(c.phi), dev(c.T) + noise(0.02 if warm else 0.0), dev(c.ux) + noise(1e-3), dev(c.uy) + noise(1e-3))


def _adjoint_inputs(case, seed):
    c = _problem(case["problem"], case["nx"], case["ny"], seed)
    c.T_wall = (0.0, 0.0, -1.0137, 0.0)
    phi, T, ux, uy = _inputs(c, seed)
    target = 0.9 * phi[0]
    return c, phi, T, ux, uy, target


def prepare(case, seed):
    if case["kind"] == "adjoint":
        c, phi, T, ux, uy, target = _adjoint_inputs(case, seed)
        return dict(case=case, c=c, s=L.Solver(c, precision="fp64"), fields=(phi, T, ux, uy), target=target)
    if case["kind"] == "batch":
        cs = _batch(case)
        fields = [_inputs(c, seed + 1000 * k) for k, c in enumerate(cs)]
        solvers = [L.Solver(c, precision=case["precision"]) for c in cs]
        for s, f in zip(solvers, fields):
            s.set_fields(*f)
        b = L.Batch(solvers).set_plan(mode=case["mode"])
        return dict(case=case, cs=cs, s=solvers, b=b, fields=fields)
    c = _problem(case["problem"], case["nx"], case["ny"], seed)
    return dict(case=case, c=c, s=L.Solver(c, precision=case["precision"]), fields=_inputs(c, seed))


def run(state):
    case = state["case"]
    if case["kind"] == "adjoint":
        phi, T, ux, uy = state["fields"]
        g = L.lbm_adjoint_fl_loss(state["s"].h, phi, T, ux, uy, state["target"], None, L.LBM_DEVICE, case["steps"],
                                  case["checkpoint"])
        n = state["c"].N
        return dict(loss=np.array([g.loss]), T_wall=np.array(list(g.T_wall)), rhoL=np.array(list(g.rhoL)[:n]),
                    lambda_s=np.array(list(g.lambda_s)[:n]), lambda_l=np.array(list(g.lambda_l)[:n]))
    dtype = _DTYPE[case["precision"]]
    if case["kind"] == "batch":
        for s, f in zip(state["s"], state["fields"]):
            s.set_fields(*f)
        state["b"].step(case["steps"])
        out = {k: [] for k in _FIELDS}
        for c, s in zip(state["cs"], state["s"]):
            F = s.fields()
            F["pcm_fl"] = pcm_liquid_fraction(c, F)
            for k in _FIELDS:
                out[k].append(F[k].reshape(-1))
        return {k: torch.cat(v).to(dtype) for k, v in out.items()}
    s = state["s"]
    s.set_fields(*state["fields"])
    s.step(case["steps"])
    F = s.fields()
    F["pcm_fl"] = pcm_liquid_fraction(state["c"], F)
    return {k: F[k].to(dtype) for k in _FIELDS}


# ---- what a pass cannot do without ----------------------------------------------------------------------

_BYTES = {"fp64": (8, 8, 8), "df64": (8, 8, 8), "fp32": (4, 4, 4), "fp16s": (4, 2, 4), "bf16s": (4, 2, 4)}
# arithmetic of one lattice update for N = 2, 3, 4 (an FMA counts two)
_FLOPS = {2: 660.0, 3: 890.0, 4: 1130.0}


def _state_bytes(N, precision):
    rest, moving, lagged = _BYTES[precision]
    return (N + 2) * rest + 8 * (N + 2) * moving + (3 + 2 * N) * lagged


def work(case):
    """Bytes: the initial fields read once, per step the state (populations and lagged values) read once and
    written once, the returned fields written once.  A gradient: the forward run, then per step the state and the
    adjoint state read and the adjoint state written."""
    K = case["steps"]
    if case["kind"] == "batch":
        cells, N = sum(c.nx * c.ny for c in _batch_sizes(case)), 2
    else:
        cells, N = case["nx"] * case["ny"], _N[case["problem"]]
    b = _state_bytes(N, case["precision"])
    if case["kind"] == "adjoint":
        return {"bytes": cells * (8 * (N + 4) + K * (2 * b + 3 * b)), "flops": cells * K * 3.0 * _FLOPS[N]}
    out = torch.empty(0, dtype=_DTYPE[case["precision"]]).element_size()
    return {"bytes": cells * (8 * (N + 3) + K * 2 * b + out * (N + 6)), "flops": cells * K * _FLOPS[N]}


class _Size:
    def __init__(self, nx, ny):
        self.nx, self.ny = nx, ny


def _batch_sizes(case):
    if case["problem"] == "sweep":
        u = W.uniform(case.get("pick", 4), 4 * case["cases"])
        sides = [W.BATCH_SIDES[min(int(u[4 * k] * len(W.BATCH_SIDES)), len(W.BATCH_SIDES) - 1)]
                 for k in range(case["cases"])]
        return [_Size(n, n) for n in sides]
    return _batch(case)


# ---- the same in 64 bits, plain torch ---------------------------------------------------------------------

_CX = (0, 1, 0, -1, 0, 1, -1, -1, 1)
_CY = (0, 0, 1, 0, -1, 1, 1, -1, -1)
_OPP = (0, 3, 4, 1, 2, 7, 8, 5, 6)
_WT = (4 / 9,) + (1 / 9,) * 4 + (1 / 36,) * 4


class _Plain:
    """The scheme of arXiv 2603.22902 (Sections 2 and 3), one full-field torch expression per quantity.  The wall
    temperatures, latent heats per volume and conductivities are tensors, so that a loss can be differentiated."""

    def __init__(self, c):
        t = lambda v: torch.tensor(v, dtype=torch.float64, device="cuda")
        col = lambda k: t([ph[k] for ph in c.phases])
        self.c, self.N = c, c.N
        self.rs, self.rl, self.ms, self.ml = col("rho_s"), col("rho_l"), col("mu_s"), col("mu_l")
        self.ls, self.ll, self.cs, self.cl = col("lam_s"), col("lam_l"), col("cp_s"), col("cp_l")
        self.rhoL = col("rho_l") * col("latent")
        self.pcm = (col("latent") > 0).double()
        self.Tw = t(list(c.T_wall))
        cp_ref = c.cp_ref if c.cp_ref > 0 else 2 * c.phases[0]["cp_s"] * c.phases[0]["cp_l"] / (
            c.phases[0]["cp_s"] + c.phases[0]["cp_l"])
        self.Eref = c.rho_ref * cp_ref
        self.sig = np.asarray(c.sigma, dtype=np.float64)
        self.wet = np.asarray(c.wet_cos, dtype=np.float64).reshape(4, c.N, c.N)

    def mix(self, a, phi):
        return (a.view(-1, 1, 1) * phi).sum(0)

    def sums(self, phi):
        rs, rl, cs, cl = (self.mix(a, phi) for a in (self.rs, self.rl, self.cs, self.cl))
        return rs, rl, cs, cl, self.mix(self.rhoL, phi)

    def enthalpy_map(self, phi, rhoH):
        c = self.c
        rs, rl, cs, cl, Lv = self.sums(phi)
        As, Al = rs * cs * c.T_sol, rl * cl * c.T_liq + Lv
        none = ~(Lv > 0)
        solid = ~none & (rhoH < As)
        liquid = none | (~solid & (rhoH > Al))
        band = ~solid & ~liquid & (Al - As > 0)
        d = torch.where(band, Al - As, torch.ones_like(Al))
        one = torch.ones_like(rhoH)
        fl = torch.where(solid, 0.0 * one, torch.where(band, (rhoH - As) / d, one))
        T = torch.where(solid, rhoH / (rs * cs),
                        torch.where(liquid, c.T_liq + (rhoH - Al) / (rl * cl),
                                    torch.where(band, c.T_sol + fl * (c.T_liq - c.T_sol), c.T_liq * one)))
        return fl, T

    def start(self, phi, T, ux, uy):
        c = self.c
        rs, rl, cs, cl, Lv = self.sums(phi)
        As, Al = rs * cs * c.T_sol, rl * cl * c.T_liq + Lv
        span = c.T_liq - c.T_sol if c.T_liq > c.T_sol else 1.0
        liquid = ~(Lv > 0) | (T >= c.T_liq)
        rhoH = torch.where(liquid, Al + rl * cl * (T - c.T_liq),
                           torch.where(T < c.T_sol, rs * cs * T, As + (T - c.T_sol) / span * (Al - As)))
        fl, T = self.enthalpy_map(phi, rhoH)
        fs = 1 - fl
        rho, cp = fs * rs + fl * rl, fs * cs + fl * cl
        uu, E = ux * ux + uy * uy, self.Eref * T
        f, g, h = [], [], []
        for i in range(9):
            cu = _CX[i] * ux + _CY[i] * uy
            s = 3 * cu + 4.5 * cu * cu - 1.5 * uu
            f.append(_WT[i] * rho * s)
            h.append(rhoH - E + _WT[0] * (E - 1.5 * rho * cp * T * uu) if i == 0 else _WT[i] * (E + rho * cp * T * s))
            g.append(_WT[i] * phi * (1 + 3 * cu))
        zero = torch.zeros_like(T)
        self.st = (torch.stack(f), torch.stack(g, 1), torch.stack(h), zero, zero,
                   fs * self.mix(self.rs - self.rl, phi), phi * ux, phi * uy)

    def pad(self, a):
        """One ghost cell around the last two axes: wrapped, or the boundary cell's value."""
        c = self.c
        x = (a[..., -1:], a, a[..., :1]) if c.bc[0] == W.PERIODIC else (a[..., :1], a, a[..., -1:])
        a = torch.cat(x, -1)
        y = (a[..., -1:, :], a, a[..., :1, :]) if c.bc[2] == W.PERIODIC else (a[..., :1, :], a, a[..., -1:, :])
        return torch.cat(y, -2)

    def at(self, padded, i):
        """Values at x + c_i of a padded field."""
        ny, nx = self.c.ny, self.c.nx
        return padded[..., 1 + _CY[i]:1 + _CY[i] + ny, 1 + _CX[i]:1 + _CX[i] + nx]

    def pad_phi(self, phi):
        """Ghosts of phi_p beyond a wall carry its wetting condition."""
        base = self.pad(phi)
        out = base.clone()
        strips = {0: (slice(None), slice(0, 1)), 1: (slice(None), slice(-1, None)),
                  2: (slice(0, 1), slice(None)), 3: (slice(-1, None), slice(None))}
        for side, (sy, sx) in strips.items():
            if self.c.bc[side] != W.WALL or not np.any(self.wet[side]):
                continue
            b = base[:, sy, sx]
            for p in range(self.N):
                corr = sum(4.0 / self.c.eps * self.wet[side, p, q] * b[p] * b[q] for q in range(self.N) if q != p)
                out[p, sy, sx] = out[p, sy, sx] + corr
        return out

    def grad(self, padded):
        v = [self.at(padded, i) for i in range(9)]
        gx = 3 * sum(_WT[i] * _CX[i] * v[i] for i in range(1, 9) if _CX[i])
        gy = 3 * sum(_WT[i] * _CY[i] * v[i] for i in range(1, 9) if _CY[i])
        return gx, gy, v

    def macro(self):
        """The macroscopic fields of the current state and what the collisions need."""
        c, N = self.c, self.N
        f, g, h, md, Qm, psim, pux, puy = self.st
        phi = g.sum(1) / (1 - 0.5 * md)
        rhoH = h.sum(0) + 0.5 * Qm
        fl, T = self.enthalpy_map(phi, rhoH)
        fs = 1 - fl
        two = lambda s, l: fs * self.mix(s, phi) + fl * self.mix(l, phi)
        rho, mu, lam, cp = two(self.rs, self.rl), two(self.ms, self.ml), two(self.ls, self.ll), two(self.cs, self.cl)
        psi, chi = fs * self.mix(self.rs - self.rl, phi), fs * self.mix(self.pcm, phi)
        gx, gy, v = self.grad(self.pad_phi(phi))
        lap = 6 * sum(_WT[i] * (v[i] - v[0]) for i in range(1, 9))
        grx, gry, _ = self.grad(self.pad(rho))
        gsx, gsy, _ = self.grad(self.pad(psi))
        gp = lambda x: 2 * x * (1 - x) * (1 - 2 * x)
        Rx, Ry = [0.0] * N, [0.0] * N
        mup = [0.0] * N
        for p in range(N):
            for q in range(p + 1, N):
                s = phi[p] + phi[q]
                Gx, Gy = phi[q] * gx[p] - phi[p] * gx[q], phi[q] * gy[p] - phi[p] * gy[q]
                G2 = Gx * Gx + Gy * Gy
                ok = (s > 1e-12) & (G2 > 1e-24 * (s * s) * (s * s))
                r = torch.where(ok, torch.where(ok, G2, torch.ones_like(G2)).rsqrt(), torch.zeros_like(G2))
                nx, ny = Gx * r, Gy * r
                a = 4.0 / c.eps * phi[p] * phi[q]
                # a derivative is not followed through the normal where it is ill-conditioned (far tails)
                fixed = (a * r).abs() > 10.0
                nx, ny = torch.where(fixed, nx.detach(), nx), torch.where(fixed, ny.detach(), ny)
                Rx[p], Ry[p], Rx[q], Ry[q] = Rx[p] + a * nx, Ry[p] + a * ny, Rx[q] - a * nx, Ry[q] - a * ny
                sg = self.sig[p, q]
                mup[p] = mup[p] + 6 * sg / c.eps * (gp(phi[p]) - gp(s)) + 0.75 * c.eps * sg * lap[q]
                mup[q] = mup[q] + 6 * sg / c.eps * (gp(phi[q]) - gp(s)) + 0.75 * c.eps * sg * lap[p]
        Fx = rho * c.accel[0] + sum(mup[p] * gx[p] for p in range(N))
        Fy = rho * c.accel[1] + sum(mup[p] * gy[p] for p in range(N))
        jx = sum(_CX[i] * f[i] for i in range(9) if _CX[i])
        jy = sum(_CY[i] * f[i] for i in range(9) if _CY[i])
        usx, usy = (jx + 0.5 * Fx) / rho, (jy + 0.5 * Fy) / rho
        fpx, fpy = chi * (c.u_solid[0] - usx), chi * (c.u_solid[1] - usy)
        ux, uy = usx + 0.5 * fpx, usy + 0.5 * fpy
        mdot = -((psi - psim) + (ux * gsx + uy * gsy)) / rho
        S = rho * mdot + (ux * grx + uy * gry)
        Lxx, Lyy, Lxy = 2 * ux * Fx + S / 3, 2 * uy * Fy + S / 3, ux * Fy + uy * Fx
        tau_f = 3 * mu / rho + 0.5
        Gx, Gy = Fx + rho * fpx, Fy + rho * fpy

        def force(i):
            q = (_CX[i] ** 2 - 1 / 3) * Lxx + 2 * _CX[i] * _CY[i] * Lxy + (_CY[i] ** 2 - 1 / 3) * Lyy
            return _WT[i] * (S + 3 * (_CX[i] * Gx + _CY[i] * Gy) + 4.5 * q)

        uu = ux * ux + uy * uy
        p = 0.6 * (f[1:].sum(0) + 0.5 * S + (tau_f - 0.5) * force(0) - rho * _WT[0] * 1.5 * uu)
        return locals()

    def step(self):
        c, N = self.c, self.N
        m = self.macro()
        f, g, h, md, Qm, psim, pux, puy = self.st
        phi, ux, uy, uu, rho, T, cp, mdot = (m[k] for k in ("phi", "ux", "uy", "uu", "rho", "T", "cp", "mdot"))
        E, Z = self.Eref * T, rho * cp * T
        tau_h = 3 * m["lam"] / self.Eref + 0.5
        tau_f, tau_g = m["tau_f"], 3 * c.mobility + 0.5
        of, og, oh = 1 / tau_f, 1 / tau_g, 1 / tau_h
        Rx, Ry = torch.stack(m["Rx"]), torch.stack(m["Ry"])
        dtx, dty = phi * ux - pux, phi * uy - puy
        fp, gpp, hp, heq = [], [], [], []
        for i in range(9):
            cu = _CX[i] * ux + _CY[i] * uy
            s = 3 * cu + 4.5 * cu * cu - 1.5 * uu
            feq = 3 * m["p"] * (_WT[i] - (1.0 if i == 0 else 0.0)) + rho * _WT[i] * s
            fp.append(f[i] - (f[i] - feq) * of + (1 - 0.5 * of) * m["force"](i))
            geq = _WT[i] * phi * (1 + 3 * cu)
            G = _WT[i] * (3 * (_CX[i] * dtx + _CY[i] * dty) + (_CX[i] * Rx + _CY[i] * Ry)) + _WT[i] * phi * mdot
            gpp.append(g[:, i] - (g[:, i] - geq) * og + (1 - 0.5 * og) * G)
            he = m["rhoH"] - E + _WT[0] * (E - 1.5 * Z * uu) if i == 0 else _WT[i] * (E + Z * s)
            heq.append(he)
            hp.append(h[i] - (h[i] - he) * oh + (1 - 0.5 * oh) * _WT[i] * Z * mdot)
        ghost = {}
        for side, row, up in ((2, 0, 1), (3, c.ny - 1, -1)):
            if c.bc[side] == W.WALL and c.tbc[side] == W.DIRICHLET:
                Eg = self.Eref * (2 * self.Tw[side] - T[row])
                for i in range(9):
                    if _CY[i] == up:
                        ghost[i] = _WT[i] * Eg + (1 - oh[row]) * (h[i][row] - heq[i][row])

        def stream(post, is_h):
            out = []
            for i in range(9):
                a = self.at(self.pad(post[i]), _OPP[i]).clone()
                for side, row, up in ((2, 0, 1), (3, c.ny - 1, -1)):
                    if _CY[i] != up or c.bc[side] != W.WALL:
                        continue
                    if is_h and c.tbc[side] == W.DIRICHLET:
                        gx = ghost[i]
                        a[..., row, :] = torch.roll(gx, _CX[i], -1) if _CX[i] else gx
                    else:
                        a[..., row, :] = post[_OPP[i]][..., row, :]
                for colx, right in ((0, 1), (c.nx - 1, -1)):
                    if _CX[i] == right and c.bc[0] != W.PERIODIC:
                        a[..., colx] = post[_OPP[i]][..., colx]
                out.append(a)
            return out

        self.st = (torch.stack(stream(fp, False)), torch.stack(stream(gpp, False), 1), torch.stack(stream(hp, True)),
                   mdot, Z * mdot, m["psi"], phi * ux, phi * uy)

    def fields(self):
        m = self.macro()
        out = {k: m[k] for k in ("phi", "T", "ux", "uy", "p")}
        out["H"] = m["rhoH"] / m["rho"]
        out["pcm_fl"] = self.mix(self.pcm, m["phi"]) * m["fl"]
        return out


def exact(case, seed):
    if case["kind"] == "adjoint":
        c, phi, T, ux, uy, target = _adjoint_inputs(case, seed)
        if c.nx * c.ny * case["steps"] > 2_000_000:
            return None
        s = _Plain(c)
        leaves = [s.Tw, s.rhoL, s.ls, s.ll]
        for v in leaves:
            v.requires_grad_(True)
        s.start(phi, T, ux, uy)
        for _ in range(case["steps"]):
            s.step()
        m = s.macro()
        loss = (s.mix(s.pcm, m["phi"]) * m["fl"] - target).square().sum()
        gr = torch.autograd.grad(loss, leaves)
        num = lambda v: v.detach().cpu().numpy()
        return dict(loss=num(loss).reshape(1), T_wall=num(gr[0]), rhoL=num(gr[1]), lambda_s=num(gr[2]),
                    lambda_l=num(gr[3]))
    with torch.no_grad():
        if case["kind"] == "batch":
            out = {k: [] for k in _FIELDS}
            for k, c in enumerate(_batch(case)):
                s = _Plain(c)
                s.start(*_inputs(c, seed + 1000 * k))
                for _ in range(case["steps"]):
                    s.step()
                F = s.fields()
                for name in _FIELDS:
                    out[name].append(F[name].reshape(-1))
            return {k: torch.cat(v) for k, v in out.items()}
        c = _problem(case["problem"], case["nx"], case["ny"], seed)
        s = _Plain(c)
        s.start(*_inputs(c, seed))
        for _ in range(case["steps"]):
            s.step()
        return s.fields()
