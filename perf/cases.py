"""Performance cases: the work that users of this package have it do, through its public
entry points, over the sizes, storage types and options they use.

Single problems go through ``lbm.Solver`` (start fields and porosity in hand, then time
steps and the macroscopic fields), sweeps through ``lbm.Batch``, the learned warm start
through ``fno.make_fno``.  ``exact`` restates each of them in plain FP64 torch.
"""
from __future__ import annotations

import math

import numpy as np
import torch
import torch.nn.functional as nnf

from paper_1409_5929_gb300 import fno, inputs, lbm

DEV = "cuda"
LISTED_WORK = 4096 * 8192 * 10   # node updates of the largest listed case

# Flow problems: the porous annulus of Fig. 3 (walls all round) with the sweep's middle
# parameters, the free-fluid annulus of Table 2, and the pipe with inlet and outlet (Fig. 1).
ANNULUS = dict(geometry=lbm.LBM_ANNULUS, Pr=0.71, eps_mean=0.6, radius_ratio=2.0)
FREE = dict(geometry=lbm.LBM_ANNULUS, Pr=0.7, eps_mean=1.0, radius_ratio=2.0, F_eps=0.0, Da=1e8)
PIPE = dict(geometry=lbm.LBM_PIPE_INFLOW, Pr=0.7, eps_mean=1.0, F_eps=0.0, Ra=0.0, Da=1e-2, tau_nu=0.6215, u_in=0.05)


def listed():
    return [
        # the smallest call: one step of the plain 48 x 96 problem, its fields read back
        dict(name="step_48x96_f32", kind="flow", flow="annulus", nr=48, nz=96, storage="f32", steps=1, Ra=1e3, Da=1e-2),
        # the plain method's run of the same problem, a stretch between two looks at it
        dict(name="run_48x96_f32", kind="flow", flow="annulus", nr=48, nz=96, storage="f32", steps=200, Ra=1e3, Da=1e-2),
        # Table 2's free-fluid annulus
        dict(name="table2_100x200_f32", kind="flow", flow="free", nr=100, nz=200, storage="f32", steps=200, Ra=1e4, Da=0.0),
        # the discretely heated annulus' and the drift test's middle grids: everything in L2
        dict(name="annulus_512x1024_f32", kind="flow", flow="annulus", nr=512, nz=1024, storage="f32", steps=50, Ra=1e5,
             Da=1e-3),
        # the benchmark's single large domain, FP32 and 16-bit storage
        dict(name="domain_4096x8192_f32", kind="flow", flow="annulus", nr=4096, nz=8192, storage="f32", steps=10, Ra=1e6,
             Da=1e-4),
        dict(name="domain_4096x8192_f16", kind="flow", flow="annulus", nr=4096, nz=8192, storage="f16", steps=10, Ra=1e6,
             Da=1e-4),
        # odd row length in BF16: no aligned pairs
        dict(name="odd_1023x2047_bf16", kind="flow", flow="annulus", nr=1023, nz=2047, storage="bf16", steps=20, Ra=1e6,
             Da=1e-3),
        # one state buffer (in-place storage), for domains that would not fit otherwise
        dict(name="inplace_2048x4096_f32", kind="flow", flow="annulus", nr=2048, nz=4096, storage="f32", steps=10, Ra=1e6,
             Da=1e-4, inplace=1),
        # part of the parameter sweep: uneven instances stepped together
        dict(name="sweep_64_f16", kind="sweep", n=64, nr_lo=64, nr_hi=512, storage="f16", steps=40, check=0),
        # small instances run towards their steady state, residual checked on the way
        dict(name="steady_16_f32", kind="sweep", n=16, nr_lo=64, nr_hi=160, storage="f32", steps=200, check=100),
        # the warm-start network at the study's size: one training step, one prediction
        dict(name="fno_train_8x128x256", kind="fno", batch=8, nr=128, nz=256, train=True),
        dict(name="fno_predict_8x64x128", kind="fno", batch=8, nr=64, nz=128, train=False),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["flow", "flow", "flow", "flow", "sweep", "fno"])
    if kind == "fno":
        nr, nz = rng.choice([(64, 128), (128, 128), (128, 256)])
        return dict(kind="fno", batch=rng.choice([1, 2, 3, 4, 5, 6, 7]), nr=nr, nz=nz, train=rng.random() < 0.6)
    if kind == "sweep":
        lo = rng.randint(40, 120)
        steady = rng.random() < 0.5
        return dict(kind="sweep", n=rng.randint(5, 16), nr_lo=lo, nr_hi=lo + rng.randint(20, 300 if not steady else 80),
                    storage=rng.choice(["f32", "f16", "bf16"]), steps=2 * rng.randint(20, 60), check=20 if steady else 0)
    flow = rng.choice(["annulus", "annulus", "annulus", "free", "pipe"])
    nr, nz = _log_int(rng, 24, 3000), _log_int(rng, 48, 6000)
    steps = max(1, min(rng.randint(2, 200), LISTED_WORK // (2 * nr * nz), 40_000_000 // (nr * nz) + 20))
    return dict(kind="flow", flow=flow, nr=nr, nz=nz, storage=rng.choice(["f32", "f32", "f16", "bf16"]), steps=steps,
                Ra=0.0 if flow == "pipe" else float("%.3g" % (nr * nr * 10 ** rng.uniform(-1.0, 0.7))),
                Da=0.0 if flow != "annulus" else float("%.3g" % 10 ** rng.uniform(-4, -1)),
                inplace=int(rng.random() < 0.2))


# ------------------------------------------------------------------ inputs --
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _smooth(nr, nz, cell, gen):
    """Standardised smooth random field: noise on a grid `cell` times coarser, bicubic."""
    a = torch.randn((1, 1, max(4, nr // cell + 2), max(4, nz // cell + 2)), device=DEV, generator=gen)
    a = nnf.interpolate(a, size=(nr, nz), mode="bicubic", align_corners=True)[0, 0]
    return a / a.abs().max()


def _fields(nr, nz, T_hot, T_cold, u_in, gen):
    """Start fields: a conduction-like temperature with a smooth disturbance and a vortex
    that vanishes at the walls (on top of the inlet velocity for the pipe)."""
    r = torch.linspace(0, 1, nr, device=DEV)[:, None]
    z = torch.linspace(0, 1, nz, device=DEV)[None, :]
    env = torch.sin(math.pi * r) * torch.sin(math.pi * z)
    amp, s = 0.02 + 0.01 * torch.rand(4, device=DEV, generator=gen), _smooth(nr, nz, max(8, nr // 6), gen)
    ur = -amp[0] * torch.sin(math.pi * r) ** 2 * torch.sin(2 * math.pi * z) + 0.2 * amp[1] * env * s
    uz = u_in + amp[0] * torch.sin(2 * math.pi * r) * torch.sin(math.pi * z) ** 2 + 0.2 * amp[2] * env * s
    T = T_hot + (T_cold - T_hot) * r + (3 * amp[3] * env * s) * (T_hot - T_cold)
    return ur.contiguous(), uz.contiguous(), T.expand(nr, nz).contiguous()


def _flow_inputs(case, seed):
    nr, nz = case["nr"], case["nz"]
    kw = dict({"annulus": ANNULUS, "free": FREE, "pipe": PIPE}[case["flow"]])
    if case["flow"] != "pipe":
        kw["Ra"] = case["Ra"]
    if case["flow"] == "annulus":
        kw["Da"] = case["Da"]
    gen = _gen(seed)
    phi = torch.ones((nr, nz), device=DEV)
    if case["flow"] == "annulus":
        phi = (0.6 + 0.28 * _smooth(nr, nz, 16, gen)).contiguous()
    return kw, phi, _fields(nr, nz, 1.0, 0.0, kw.get("u_in", 0.0), gen)


def _sweep_inputs(case, seed):
    inst = inputs.sweep_instances(case["n"], seed=int(seed) % (1 << 31), nr_lo=case["nr_lo"], nr_hi=case["nr_hi"])
    # the sizes are the case's own, the same for every seed
    sizes = np.random.default_rng(case["n"] * 1009 + case["nr_lo"]).integers(case["nr_lo"], case["nr_hi"] + 1, case["n"])
    gen = _gen(seed)
    out = []
    for d, nr in zip(inst, sizes):
        nr = int(nr)
        kw = dict(geometry=lbm.LBM_ANNULUS, Ra=d["Ra"], Da=d["Da"], Pr=d["Pr"], eps_mean=d["eps"],
                  radius_ratio=d["radius_ratio"])
        out.append((nr, 2 * nr, kw, _fields(nr, 2 * nr, 1.0, 0.0, 0.0, gen)))
    return out


def _fno_inputs(case, seed):
    """Network inputs and targets with the ranges of the warm start's features."""
    b, nr, nz = case["batch"], case["nr"], case["nz"]
    gen = _gen(seed)
    x = torch.empty((b, nr, nz, 8), device=DEV)
    t = torch.empty((b, nr, nz, 3), device=DEV)
    par = 2 * torch.rand((b, 5), device=DEV, generator=gen) - 1
    for i in range(b):
        x[i, :, :, 0] = par[i, 2] + 0.4 * _smooth(nr, nz, 8, gen)
        x[i, :, :, 1:6] = par[i]
        ur, uz, T = _fields(nr, nz, 1.0, 0.0, 0.0, gen)
        t[i] = torch.stack([ur * 17.3, uz * 17.3, 2 * (T - 0.5)], dim=-1)
    x[..., 6] = torch.linspace(-1, 1, nr, device=DEV)[:, None]
    x[..., 7] = torch.linspace(-1, 1, nz, device=DEV)[None, :]
    # weights as a network starts from: width 32, 16 modes, hidden 128
    rng, P = np.random.default_rng(seed), {}

    def lin(i, o, w, b):
        a = 1.0 / math.sqrt(i)
        P[w], P[b] = ((2 * a * rng.random(s, dtype=np.float32) - a).astype(np.float32) for s in ((i, o), (o,)))

    lin(8, 32, "P", "p")
    for l in range(4):
        P[f"R{l}"] = rng.random((32, 16, 32, 32, 2), dtype=np.float32) / np.float32(32 * 32)
        lin(32, 32, f"W{l}", f"b{l}")
    lin(32, 128, "Q1", "q1")
    lin(128, 3, "Q2", "q2")
    return x, t, P


# --------------------------------------------------------------- the cases --
def prepare(case, seed):
    if case["kind"] == "flow":
        kw, phi, (ur, uz, T) = _flow_inputs(case, seed)
        s = lbm.Solver(nr=case["nr"], nz=case["nz"], storage=case["storage"], inplace=case.get("inplace", 0), **kw)
        s.set_porosity(phi)
        s.init_fields(ur, uz, T)
        return dict(case=case, s=s, out=[torch.empty_like(phi) for _ in range(4)])
    if case["kind"] == "sweep":
        inst = _sweep_inputs(case, seed)
        b = lbm.Batch([lbm.lbm_params_default(nr=nr, nz=nz, storage=case["storage"], **kw) for nr, nz, kw, _ in inst])
        torch.cuda.synchronize()   # the batch works on its own stream
        for i, (_, _, _, (ur, uz, T)) in enumerate(inst):
            lbm.lbm_batch_init_fields(b.b, i, ur, uz, T, True)
        sizes = [nr * nz for nr, nz, _, _ in inst]
        return dict(case=case, b=b, sizes=sizes, out=[torch.empty(sum(sizes), device=DEV) for _ in range(4)])
    x, t, weights = _fno_inputs(case, seed)
    net = fno.make_fno(case["nr"], case["nz"], params=weights)
    return dict(case=case, net=net, x=x, t=t)


def run(state):
    case = state["case"]
    if case["kind"] == "flow":
        s = state["s"]
        s.step(case["steps"])
        lbm.lbm_moments(s.h, *state["out"], True)
        return state["out"]
    if case["kind"] == "sweep":
        b = state["b"]
        if case["check"]:
            b.run(case["steps"], case["check"], -1.0)
        else:
            b.step(case["steps"])
        at = 0
        for i, n in enumerate(state["sizes"]):
            lbm.lbm_batch_moments(b.b, i, *[o[at:at + n] for o in state["out"]], True)
            at += n
        return state["out"]
    net = state["net"]
    if not case["train"]:
        return net.forward(state["x"])
    net.zero_grad()
    loss = net.loss_and_grad(state["x"], state["t"])
    return {"loss": loss, "grads": net.g}


# Operations of one node update, counted on the formulas (Eq. 6-8, 21-30, 33-38).
FLOPS_NODE = 330


def work(case):
    if case["kind"] == "fno":
        px, w, m, hid = case["batch"] * case["nr"] * case["nz"], 32, 16, 128
        nr, nz, b = case["nr"], case["nz"], case["batch"]
        spectral = 2 * b * w * (2 * m * nr * nz + 2 * 4 * m * nr * 2 * m) + 8 * b * 2 * m * m * w * w // 2
        fwd = 2 * px * (8 * w + 4 * w * w + w * hid + hid * 3) + 4 * 2 * spectral
        weights = 4 * (4 * 2 * m * m * w * w * 2 + 4 * w * w + 8 * w + w * hid + hid * 3)
        if case["train"]:
            return {"bytes": px * (8 + 3) * 4 + 2 * weights, "flops": 3 * fwd}
        return {"bytes": px * (8 + 3) * 4 + weights, "flops": fwd}
    if case["kind"] == "sweep":
        sizes = np.random.default_rng(case["n"] * 1009 + case["nr_lo"]).integers(case["nr_lo"], case["nr_hi"] + 1, case["n"])
        nodes = int(sum(2 * int(n) * int(n) for n in sizes))
    else:
        nodes = case["nr"] * case["nz"]
    pop = 14 * 4 if case["storage"] == "f32" else 9 * 2 + 5 * 4
    ref = 2 if case["storage"] == "f32" else 8
    # the state read and written once, porosity and references read, four fields written
    return {"bytes": nodes * (2 * pop + 4 + ref + 16), "flops": nodes * FLOPS_NODE * case["steps"]}


# ------------------------------------------------- the same in plain FP64 --
ER = (0, 1, 0, -1, 0, 1, -1, -1, 1)
EZ = (0, 0, 1, 0, -1, 1, 1, -1, -1)
W9 = (4 / 9,) + (1 / 9,) * 4 + (1 / 36,) * 4
W5 = (0.6, 0.1, 0.1, 0.1, 0.1)
CS2 = 1.0 / 3.0
M9 = np.array([[1, 1, 1, 1, 1, 1, 1, 1, 1], [-4, -1, -1, -1, -1, 2, 2, 2, 2], [4, -2, -2, -2, -2, 1, 1, 1, 1],
               ER, [0, -2, 0, 2, 0, 1, -1, -1, 1], EZ, [0, 0, -2, 0, 2, 1, 1, -1, -1],
               [0, 1, -1, 1, -1, 0, 0, 0, 0], [0, 0, 0, 0, 0, 1, -1, 1, -1]], dtype=np.float64)
MI9 = M9.T / (M9 ** 2).sum(axis=1)[None, :]


class _Lattice:
    """One problem of Eq. 6-42 in FP64, whole populations f (factor r) and g."""

    def __init__(self, nr, nz, kw, phi, ur, uz, T):
        p = dict(Ra=1e3, Da=1e-2, Pr=1.0, Ma=0.1, tau_nu=0.0, F_eps=-1.0, eps_mean=0.6, radius_ratio=2.0, u_in=0.0)
        p.update(kw)
        self.nr, self.nz, self.pipe = nr, nz, p["geometry"] == lbm.LBM_PIPE_INFLOW
        L = nr - 0.5 if self.pipe else nr - 1.0
        r0 = 0.5 if self.pipe else L / (p["radius_ratio"] - 1)
        cs = math.sqrt(CS2)
        if p["tau_nu"] > 0:
            tau, Ma = p["tau_nu"], 0.0
        else:
            Ma = p["Ma"]
            tau = 0.5 + Ma * L * math.sqrt(p["Pr"]) / (cs * math.sqrt(p["Ra"]))
        nu = CS2 * (tau - 0.5)
        self.tau, self.nu = tau, nu
        self.tauT = CS2 * (tau - 0.5) / (0.2 * p["Pr"])
        self.gb = (Ma * cs) ** 2 / L if p["Ra"] > 0 else 0.0
        self.u_in = p["u_in"]
        self.r = (r0 + torch.arange(nr, device=DEV, dtype=torch.float64))[:, None]
        self.phi = phi.double()
        K, em = p["Da"] * L * L, p["eps_mean"]
        if em >= 1:
            self.lin = torch.full((1, 1), nu / K, device=DEV, dtype=torch.float64)
            self.nl = (1.75 / math.sqrt(150 * K)) * self.phi ** -1.5 if p["F_eps"] < 0 else torch.zeros_like(self.lin)
        else:
            ck = em ** 3 / ((1 - em) ** 2 * K)
            self.lin = nu * ck * (1 - self.phi) ** 2 / self.phi ** 3
            self.nl = 1.75 * math.sqrt(ck / 150) * (1 - self.phi) / self.phi ** 3
        self._walls()
        self._start(ur.double(), uz.double(), T.double())

    def _walls(self):
        nr, nz = self.nr, self.nz
        kr, kz = torch.meshgrid(torch.arange(nr, device=DEV), torch.arange(nz, device=DEV), indexing="ij")
        end = (kz == 0) | (kz == nz - 1)
        wall = (kr == nr - 1) | end | ((kr == 0) & (not self.pipe))
        self.wi = wall.reshape(-1).nonzero()[:, 0]
        kr, kz = kr.reshape(-1)[self.wi], kz.reshape(-1)[self.wi]
        fr = kr.clamp(0 if self.pipe else 1, nr - 2)
        fz = kz.clamp(1, nz - 2)
        self.fi = fr * nz + fz
        self.rb, self.rf = self.r[kr, 0], self.r[fr, 0]
        hot, cold = (kz == 0, (kr == nr - 1) & ~((kz == 0) | (kz == nz - 1))) if self.pipe else (kr == 0, kr == nr - 1)
        self.hot, self.cold = hot, cold
        self.out = (kz == nz - 1) if self.pipe else torch.zeros_like(hot)

    def _wall_T(self, Tf):
        return torch.where(self.hot, torch.ones_like(Tf), torch.where(self.cold, torch.zeros_like(Tf), Tf))

    def _start(self, ur, uz, T):
        ur, uz, T = ur.clone().reshape(-1), uz.clone().reshape(-1), T.clone().reshape(-1)
        T[self.wi] = self._wall_T(T[self.fi])
        ur[self.wi] = 0.0
        uz[self.wi] = torch.where(self.hot, self.u_in, 0.0).double() if self.pipe else 0.0
        ur, uz, T = (a.reshape(self.nr, self.nz) for a in (ur, uz, T))
        rho = torch.ones_like(T)
        me, S = self._meq(rho, ur, uz), self._source(rho, ur, uz, T)
        self.f = torch.stack([sum(MI9[i, k] * (me[k] - 0.5 * S[k]) for k in range(9) if MI9[i, k]) for i in range(9)])
        self.g = torch.stack([self._geq(i, T, ur, uz) for i in range(5)])
        keep = ur.reshape(-1)[self.wi], uz.reshape(-1)[self.wi]
        self._recover()
        self.ur.reshape(-1)[self.wi], self.uz.reshape(-1)[self.wi] = keep
        self._collide()

    @staticmethod
    def _geq(i, T, ur, uz):
        return W5[i] * T * (1 + 5 * (ER[i] * ur + EZ[i] * uz))

    def _force(self, ur, uz, T):
        drag = -self.phi * (self.lin + self.nl * torch.sqrt(ur * ur + uz * uz))
        Fr = drag * ur + CS2 * (1 - 2 * (self.tau - 0.5) * ur / self.r) / self.r
        return Fr, drag * uz + self.phi * self.gb * (T - 0.5)

    def _source(self, rho, ur, uz, T):
        Fr, Fz = self._force(ur, uz, T)
        rr, ip = self.r * rho, 1 / self.phi
        a, b, c, d = ur * Fr, uz * Fz, ur * Fz, uz * Fr
        return [torch.zeros_like(a), 6 * rr * ip * (a + b), -6 * rr * ip * (a + b), rr * Fr, -rr * Fr, rr * Fz, -rr * Fz,
                2 * rr * ip * (a - b), rr * ip * (c + d)]

    def _meq(self, rho, ur, uz):
        rr, ip = self.r * rho, 1 / self.phi
        q = 3 * rr * ip * (ur * ur + uz * uz)
        return [rr, -2 * rr + q, rr - q, rr * ur, -rr * ur, rr * uz, -rr * uz, rr * ip * (ur * ur - uz * uz),
                rr * ip * ur * uz]

    def _recover(self):
        f, r, phi = self.f, self.r, self.phi
        self.T = self.g.sum(0)
        self.rho = f.sum(0) / r
        vr = (f[1] - f[3] + f[5] - f[6] + f[8] - f[7]) / self.rho + 0.5 * CS2
        vz = (f[2] - f[4] + f[5] + f[6] - f[7] - f[8]) / self.rho + 0.5 * r * phi * self.gb * (self.T - 0.5)
        hd = 0.25 * r * phi * self.lin
        x = 0.5 * r * phi * self.nl * torch.sqrt(vr * vr + vz * vz)
        lr, lz = 0.5 * (r + self.nu / r) + hd, 0.5 * r + hd
        self.ur = vr / (lr + torch.sqrt(lr * lr + x))
        self.uz = vz / (lz + torch.sqrt(lz * lz + x))

    def _collide(self):
        m = [sum(M9[k, i] * self.f[i] for i in range(9) if M9[k, i]) for k in range(9)]
        me, S = self._meq(self.rho, self.ur, self.uz), self._source(self.rho, self.ur, self.uz, self.T)
        s = (1.0, 1.1, 1.1, 1.0, 1.2, 1.0, 1.2, 1 / self.tau, 1 / self.tau)
        d = [-s[k] * (m[k] - me[k]) + (1 - 0.5 * s[k]) * S[k] for k in range(9)]
        del m, me, S
        for i in range(9):
            self.f[i] += sum(MI9[i, k] * d[k] for k in range(1, 9) if MI9[i, k])
        for i in range(5):
            om = (1 + ER[i] * self.tauT / self.r) / (self.tauT + 0.5)
            ge = self._geq(i, self.T, self.ur, self.uz)
            self.g[i] += -om * (self.g[i] - ge) - self.ur / self.r * ge

    def _stream(self):
        f0, g0 = self.f[:, 0].clone(), self.g[:, 0].clone()
        for i in range(9):
            self.f[i] = torch.roll(self.f[i], (ER[i], EZ[i]), (0, 1))
            if i < 5:
                self.g[i] = torch.roll(self.g[i], (ER[i], EZ[i]), (0, 1))
        if self.pipe:   # the axis row's inward populations come from its mirror image
            self.f[1, 0], self.f[5, 0], self.f[8, 0] = f0[3], torch.roll(f0[6], 1), torch.roll(f0[7], -1)
            self.g[1, 0] = g0[3]

    def _feq(self, i, r, rho, ur, uz, phi):
        eu = ER[i] * ur + EZ[i] * uz
        return W9[i] * r * rho * (1 + 3 * eu + 4.5 * eu * eu / phi - 1.5 * (ur * ur + uz * uz) / phi)

    def _boundary(self):
        at = lambda a, n: a.reshape(-1)[n]  # noqa: E731
        fr, fz, fT, frho, fphi = (at(a, self.fi) for a in (self.ur, self.uz, self.T, self.rho, self.phi))
        Tb, bphi = self._wall_T(fT), at(self.phi, self.wi)
        if self.pipe:
            ur = torch.where(self.out, fr, 0.0)
            uz = torch.where(self.out, fz, torch.where(self.hot, self.u_in, 0.0))
            rho = torch.where(self.out, 1.0, frho)
        else:
            ur, uz, rho = torch.zeros_like(fr), torch.zeros_like(fr), frho
        tot = 0.0
        for i in range(9):
            v = self._feq(i, self.rb, rho, ur, uz, bphi) + at(self.f[i], self.fi) - self._feq(i, self.rf, frho, fr, fz, fphi)
            self.f[i].view(-1)[self.wi] = v
            tot = tot + v
        for i in range(5):
            v = self._geq(i, Tb, ur, uz) + at(self.g[i], self.fi) - self._geq(i, fT, fr, fz)
            self.g[i].view(-1)[self.wi] = v
        for a, v in ((self.ur, ur), (self.uz, uz), (self.T, Tb), (self.rho, tot / self.rb)):
            a.view(-1)[self.wi] = v

    def _pull(self):
        self._stream()
        self._recover()
        self._boundary()

    def after(self, steps):
        for _ in range(steps):
            self._pull()
            self._collide()
        self._pull()
        return [self.rho, self.ur, self.uz, self.T]


def _net(P, x, m=16, layers=4):
    """The operator in FP64: spectral layers by rfft2 with the retained modes."""
    nr, nz = x.shape[1:3]
    h = x @ P["P"] + P["p"]
    for l in range(layers):
        R = torch.complex(P[f"R{l}"][..., 0], P[f"R{l}"][..., 1])
        X = torch.fft.rfft2(h.permute(0, 3, 1, 2))
        Y = torch.zeros(X.shape[0], R.shape[-1], nr, nz // 2 + 1, dtype=X.dtype, device=X.device)
        kr = list(range(m)) + list(range(nr - m, nr))
        Y[:, :, kr, :m] = torch.einsum("bcxy,xyco->boxy", X[:, :, kr, :m], R)
        h = h @ P[f"W{l}"] + P[f"b{l}"] + torch.fft.irfft2(Y, s=(nr, nz)).permute(0, 2, 3, 1)
        h = nnf.gelu(h) if l < layers - 1 else h
    return nnf.gelu(h @ P["Q1"] + P["q1"]) @ P["Q2"] + P["q2"]


def exact(case, seed):
    if case["kind"] == "flow":
        kw, phi, (ur, uz, T) = _flow_inputs(case, seed)
        return _Lattice(case["nr"], case["nz"], kw, phi, ur, uz, T).after(case["steps"])
    if case["kind"] == "sweep":
        parts = []
        for nr, nz, kw, (ur, uz, T) in _sweep_inputs(case, seed):
            phi = torch.full((nr, nz), float(np.float32(kw["eps_mean"])), device=DEV)
            parts.append([a.reshape(-1) for a in _Lattice(nr, nz, kw, phi, ur, uz, T).after(case["steps"])])
        return [torch.cat([q[k] for q in parts]) for k in range(4)]
    x, t, weights = _fno_inputs(case, seed)
    x, t = x.double(), t.double()
    P = {k: torch.tensor(v, dtype=torch.float64, device=DEV, requires_grad=case["train"]) for k, v in weights.items()}
    y = _net(P, x)
    if not case["train"]:
        return y
    loss = ((y - t) ** 2).mean()
    loss.backward()
    return {"loss": loss.detach().reshape(1), "grads": {k: v.grad for k, v in P.items()}}
