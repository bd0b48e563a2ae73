"""The work a user of the reservoir solver has it do, as measurable cases.

Four kinds of work, all through the package's public entry points:

* "step":   a simulator continues a run from a saved state: the state goes in
            (set_state, device buffers), one time step is advanced, the new
            state comes out (get_state).  This is what the framework is for;
            the benchmark reports exactly this on the 1M-cell model.
* "linsys": a caller's own Newton system: values, right-hand side and
            reordering key are set, the solver is set up and solves it.
* "batch":  an ensemble of independent models takes one time step.
* "train" / "predict": the learned warm start's network, one training step
            (gradients and updated weights) or one prediction.

Models are the package's own synthetic workloads (inputs.case0, case1, case2
and the ensemble's members); the seed draws the geology.  The 64-bit
reference (exact) is a plain torch restatement of the discretised equations
solved with dense linear algebra, and of the network with autograd.
"""
import math
import os

import numpy as np
import torch

import paper_1701_06254_gb300 as R
from paper_1701_06254_gb300 import inputs as I

DEV = "cuda" if torch.cuda.is_available() else "cpu"
PREC = {"fp64": R.PREC_FP64, "mixed": R.PREC_MIXED, "mixed_bf16": R.PREC_MIXED_BF16}
DEC = {"abf": R.DEC_ABF, "qi": R.DEC_QI, "none": R.DEC_NONE}
KRYLOV = {"fgmres": R.KRYLOV_FGMRES, "bicgstab": R.KRYLOV_BICGSTAB}
WEIGHTS = os.path.join(os.path.dirname(os.path.abspath(R.__file__)), "warm_start_64x64x16.npz")


def _step(name, model, nx, ny, nz, prec, dec="abf", krylov="fgmres", overlap=1, warm=1, learned=False):
    return dict(name=name, kind="step", model=model, nx=nx, ny=ny, nz=nz, prec=prec, dec=dec, krylov=krylov,
                overlap=overlap, warm=warm, learned=learned)


def _linsys(name, model, nx, ny, nz, prec, dec, tol):
    return dict(name=name, kind="linsys", model=model, nx=nx, ny=ny, nz=nz, prec=prec, dec=dec, tol=tol)


def listed():
    return [
        # the smallest model users run (the 2,000-cell tutorial-size case, library defaults): every launch and
        # host wait counts, the arithmetic does not
        _step("step_lognormal_2k_fp64", "lognormal", 20, 20, 5, "fp64", warm=2),
        # an ordinary field model with inexact Newton: setups weigh more than iterations
        _step("step_fivespot_200k_inexact", "fivespot", 100, 100, 20, "mixed"),
        # the benchmark's own model and configuration, the largest ordinary use
        _step("step_channelised_1m", "channelised", 200, 200, 25, "mixed_bf16", dec="qi", warm=2),
        # plain FP64 throughout on a ragged grid (no side divides by the 4x4 tiles or by 32)
        _step("step_channelised_odd_fp64", "channelised", 117, 93, 19, "fp64", dec="qi"),
        # the other Krylov method and the wider Schwarz overlap the paper uses, ragged grid
        _step("step_bicgstab_overlap2", "channelised", 90, 71, 15, "mixed", dec="qi", krylov="bicgstab", overlap=2),
        # a run with the learned initial guess, on the grid its network was trained on
        _step("step_learned_64x64x16", "channelised", 64, 64, 16, "mixed_bf16", dec="qi", learned=True),
        # callers' own Newton systems: a small one in full precision, an ordinary ragged one, and a large one
        # solved loosely, where the setup weighs most
        _linsys("linsys_1k_fp64", "lognormal", 14, 13, 7, "fp64", "abf", 1e-8),
        _linsys("linsys_155k_mixed", "channelised", 101, 73, 21, "mixed", "abf", 1e-6),
        _linsys("linsys_1m_loose", "channelised", 200, 200, 25, "mixed_bf16", "qi", 1e-4),
        # an ensemble: several models of different sizes in flight together
        dict(name="batch_8_members", kind="batch", members=8, sizes=2000, prec="mixed_bf16", dec="qi", workers=8),
        # the warm start's network: one training sample on the recorded grid, one prediction on a ragged one
        dict(name="train_64x64x16", kind="train", nx=64, ny=64, nz=16),
        dict(name="predict_97x61x23", kind="predict", nx=97, ny=61, nz=23),
    ]


def _size(rng, lo, hi):
    """Grid of about lo..hi cells (log-uniform), nz from the flat to the thick, sides not rounded."""
    cells = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    nz = max(3, min(32, int(round(math.exp(rng.uniform(math.log(0.5), math.log(2.0))) * cells ** 0.25))))
    side = math.sqrt(cells / nz)
    aspect = math.exp(rng.uniform(math.log(0.6), math.log(1.6)))
    return max(12, int(side * aspect)), max(12, int(side / aspect)), nz


def draw(rng):
    kind = rng.choice(["step"] * 5 + ["linsys"] * 3 + ["batch", "train", "predict"])
    if kind in ("step", "linsys"):
        nx, ny, nz = _size(rng, 1.5e3, 6e5)
        prec = rng.choice(["fp64", "mixed", "mixed_bf16", "mixed_bf16"])
        if prec == "fp64":
            nx, ny = min(nx, 130), min(ny, 130)
        model = rng.choice(["fivespot", "channelised", "channelised"]) if nx * ny * nz > 4000 else "lognormal"
        dec = rng.choice(["qi", "qi", "abf"]) if model == "channelised" else "abf"
        if kind == "linsys":
            c = _linsys("", model, nx, ny, nz, prec, dec, rng.choice([1e-4, 1e-6, 1e-8]))
        else:
            c = _step("", model, nx, ny, nz, prec, dec=dec, krylov=rng.choice(["fgmres", "fgmres", "bicgstab"]),
                      overlap=rng.choice([1, 1, 2]), learned=model == "channelised" and rng.random() < 0.2)
    elif kind == "batch":
        c = dict(kind="batch", members=rng.randint(2, 8), sizes=rng.randint(1, 10 ** 6), prec=rng.choice(["mixed", "mixed_bf16"]),
                 dec="qi", workers=rng.choice([2, 4, 8]))
    else:
        nx, ny, nz = _size(rng, 2e3, 3e5)
        c = dict(kind=kind, nx=nx, ny=ny, nz=nz)
    c.pop("name", None)
    return c


# ------------------------------------------------------------- inputs ------
def _geology(c, seed):
    if c["model"] == "channelised":
        return I.case2(seed=seed, nx=c["nx"], ny=c["ny"], nz=c["nz"])
    if c["model"] == "fivespot":
        return I.case1(seed=seed, nx=c["nx"], ny=c["ny"], nz=c["nz"])
    if (c["nx"], c["ny"], c["nz"]) == (20, 20, 5):
        return I.case0(seed=seed)
    return I.small_case(c["nx"], c["ny"], c["nz"], seed=seed)


def _member_sizes(c):
    """The members' grids, drawn as the ensemble workload draws them: U{32..128} x U{32..128} x U{8..32}."""
    rng = np.random.default_rng(c["sizes"])
    return [[int(rng.integers(lo, hi + 1)) for lo, hi in ((32, 128), (32, 128), (8, 32))] for _ in range(c["members"])]


def _options(c):
    o = dict(precision=PREC[c["prec"]], decoupling=DEC[c["dec"]])
    if "krylov" in c:
        o.update(krylov=KRYLOV[c["krylov"]], overlap=c["overlap"])
    return o


def _state_of(sim):
    p, sw, pb, t = sim.get_state()
    return [torch.from_numpy(a).to(DEV) for a in (p, sw, pb)], t


def _like(state):
    return [torch.empty_like(a) for a in state]


def _features(c, seed):
    """Network inputs as a run gives them: smooth fields of unit rms concentrated around a few wells, plus the
    piecewise ln k; the last two channels are zero."""
    rng = np.random.default_rng(seed)
    nz, ny, nx = c["nz"], c["ny"], c["nx"]
    z, y, x = np.meshgrid(np.linspace(0, 1, nz), np.linspace(0, 1, ny), np.linspace(0, 1, nx), indexing="ij")
    f = np.zeros((nz, ny, nx, 8))
    for ch in (0, 1, 4, 5, 6, 7):
        for _ in range(6):
            w = rng.uniform(0.05, 0.3)
            r2 = ((x - rng.random()) ** 2 + (y - rng.random()) ** 2 + 0.3 * (z - rng.random()) ** 2) / (w * w)
            f[..., ch] += rng.standard_normal() * np.exp(-r2)
        f[..., ch] += 0.05 * rng.standard_normal((nz, ny, nx))
        f[..., ch] /= np.sqrt(np.mean(f[..., ch] ** 2))
    target = np.ascontiguousarray(f[..., 6:8]).astype(np.float32)
    f[..., 2] = 0.5 * (np.where(rng.random((nz, ny, nx)) < 0.35, math.log(500.0), math.log(5.0)) - 4.0)
    f[..., 3] = 4.0 * (0.2 + 0.3 * np.abs(f[..., 5]) / (1.0 + np.abs(f[..., 5])) - 0.5)
    f[..., 6:8] = 0.0
    return f.astype(np.float32), target


def _weights(c, seed):
    """The trained weights for a prediction; for training, an early network (He-normal, a small head)."""
    if c["kind"] != "train":
        return np.load(WEIGHTS, allow_pickle=False)["params"].astype(np.float32)
    rng = np.random.default_rng(seed + 5)
    flat = []
    for k, (_, ci, co) in enumerate(_LAYERS):
        scale = math.sqrt((2.0 if k + 1 < len(_LAYERS) else 0.1) / (27 * ci))
        flat += [scale * rng.standard_normal(27 * ci * co), 0.01 * rng.standard_normal(co)]
    return np.concatenate(flat).astype(np.float32)


def prepare(case, seed):
    c = case
    if c["kind"] == "step":
        sim = R.Sim(_geology(c, seed), **_options(c))
        ws = None
        if c["learned"]:
            ws = R.WarmStart()
            ws.set_params(_weights(c, seed))
            sim.attach_warm_start(ws)
        sim.init_hydrostatic()
        sim.advance(c["warm"])
        state, t = _state_of(sim)
        return dict(c=c, sim=sim, ws=ws, state=state, t=t, out=_like(state))
    if c["kind"] == "linsys":
        geo = _geology(c, seed)
        rp, ci, val, b, key = _linear_system(geo, seed)
        wc0 = np.array([w.perf_cells[0] for w in geo.wells], np.int32)
        ls = R.LinearSystem(geo.nx, geo.ny, geo.nz, len(geo.wells), rp.cpu().numpy(), ci.cpu().numpy(), wc0,
                            **_options(c))
        return dict(c=c, ls=ls, val=val, b=b, key=key, y=torch.empty_like(b))
    if c["kind"] == "batch":
        geo = [I.case2(seed=seed + 1000 * k, nx=nx, ny=ny, nz=nz) for k, (nx, ny, nz) in enumerate(_member_sizes(c))]
        b = R.Batch(geo, workers=c["workers"], **_options(c))
        b.init_hydrostatic()
        b.advance(1)
        states = [_state_of(m) for m in b.members]
        return dict(c=c, batch=b, states=states, outs=[_like(s) for s, _ in states])
    ws = R.WarmStart()
    ws.set_params(_weights(c, seed))
    feat, target = _features(c, seed)
    return dict(c=c, ws=ws, feat=feat, target=target)


def run(state):
    s, kind = state, state["c"]["kind"]
    if kind == "step":
        s["sim"].set_state(*s["state"], s["t"])
        s["sim"].advance(1)
        s["sim"].get_state(out=s["out"])
        return s["out"]
    if kind == "linsys":
        s["ls"].set(s["val"], s["b"], s["key"])
        s["ls"].setup()
        s["ls"].solve(s["c"]["tol"], y=s["y"])
        return s["y"]
    if kind == "batch":
        for m, (st, t) in zip(s["batch"].members, s["states"]):
            m.set_state(*st, t)
        s["batch"].advance(1)
        for m, out in zip(s["batch"].members, s["outs"]):
            m.get_state(out=out)
        return s["outs"]
    if kind == "train":
        s["ws"].zero_grad()
        loss = s["ws"].backward(s["feat"], s["target"])
        grad = s["ws"].params(1)
        s["ws"].adam(1e-4)
        return dict(loss=loss, grad=grad, weights=s["ws"].params(0))
    return s["ws"].forward(s["feat"])


def work(case):
    c = case
    if c["kind"] in ("train", "predict"):
        v, flops = c["nx"] * c["ny"] * c["nz"], 0.0
        n = [v]
        for _ in range(3):
            n.append(-(-n[-1] // 8))
        for level, ci, co in _LAYERS:
            flops += 2.0 * 27 * ci * co * n[level]
        params = 4.0 * _n_params()
        if c["kind"] == "train":
            return dict(bytes=4.0 * v * (8 + 2) + 5 * params, flops=3.0 * flops)
        return dict(bytes=4.0 * v * (8 + 8) + params, flops=flops)
    if c["kind"] == "batch":
        cells = float(sum(nx * ny * nz for nx, ny, nz in _member_sizes(c)))
    else:
        cells = float(c["nx"] * c["ny"] * c["nz"])
    if c["kind"] == "linsys":
        # 7 blocks of 4 doubles and their columns, b, key and y per cell; one product with the matrix
        return dict(bytes=cells * (7 * (32 + 4) + 16 + 8 + 16), flops=cells * 7 * 8)
    # state in and out, rock (three permeabilities and porosity); one residual and Jacobian
    return dict(bytes=cells * (2 * 16 + 4 * 8), flops=cells * 400)


# ----------------------------------- the discretised equations in torch ----
C_DARCY = 9.869233e-16 * 1e5 / 1e-3 * 86400.0


class _Model:
    """Two-phase flow of one inputs.Case on a 64-bit torch device (fluids without capillary pressure and with
    constant viscosity, as every case here)."""

    def __init__(self, geo):
        t = lambda a: torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device=DEV)  # noqa: E731
        self.g, self.f = geo, geo.fluid
        self.n, self.nw = geo.n, len(geo.wells)
        self.nb = self.n + self.nw
        sh = (geo.nz, geo.ny, geo.nx)
        self.shape = sh
        self.z = (geo.top + (torch.arange(geo.nz, dtype=torch.float64, device=DEV) + 0.5) * geo.dz)[:, None, None].expand(sh)
        self.gz = self.f.g * self.z * 1e-5
        self.phi = t(geo.phi).reshape(sh)
        kx, ky, kz = (t(a).reshape(sh) for a in (geo.kx, geo.ky, geo.kz))
        harm = lambda k, d, a, ax: C_DARCY * a / (d / (2.0 * k.narrow(ax, 0, k.shape[ax] - 1)) + d / (2.0 * k.narrow(ax, 1, k.shape[ax] - 1)))  # noqa: E731
        self.trans = [harm(kz, geo.dz, geo.dx * geo.dy, 0), harm(ky, geo.dy, geo.dx * geo.dz, 1),
                      harm(kx, geo.dx, geo.dy * geo.dz, 2)]
        self.idx = torch.arange(self.n, device=DEV).reshape(sh)
        self.wells = []
        for w in geo.wells:
            cells = torch.as_tensor(w.perf_cells, device=DEV)
            a, b = kx.reshape(-1)[cells], ky.reshape(-1)[cells]
            ro = 0.28 * torch.sqrt(torch.sqrt(b / a) * geo.dx ** 2 + torch.sqrt(a / b) * geo.dy ** 2) / ((b / a) ** 0.25 + (a / b) ** 0.25)
            wi = 2.0 * math.pi * C_DARCY * torch.sqrt(a * b) * geo.dz / (torch.log(ro / w.r_w) + w.skin)
            dz5 = self.f.g * (self.z.reshape(-1)[cells] - geo.well_z_ref(w)) * 1e-5
            self.wells.append((w, cells, wi, dz5))

    def hydrostatic(self):
        f, g = self.f, self.g
        pot = g.p_init - f.rho_ref[1] * (1.0 + f.c_f[1] * (g.p_init - f.p_ref)) * f.g * g.top * 1e-5
        p = (pot + f.rho_ref[1] * (1.0 - f.c_f[1] * f.p_ref) * self.gz) / (1.0 - f.rho_ref[1] * f.c_f[1] * self.gz)
        return p.contiguous(), torch.full_like(p, g.sw_init)

    def well_start(self, p):
        """p_b of a BHP well at its target, of a rate well 10 bar off its first cell."""
        pf = p.reshape(-1)
        return torch.stack([torch.as_tensor(w.target, dtype=torch.float64, device=DEV) if w.control == I.BHP
                            else pf[cells[0]] + (10.0 if w.kind == I.INJ else -10.0) for w, cells, _, _ in self.wells])

    def accumulation(self, p, s):
        f = self.f
        por = self.phi * (1.0 + f.c_r * (p - f.p_ref))
        rho = [f.rho_ref[a] * (1.0 + f.c_f[a] * (p - f.p_ref)) for a in (0, 1)]
        return por * rho[1] * (1.0 - s), por * rho[0] * s

    def key(self, p):
        f = self.f
        return (p - f.rho_ref[1] * (1.0 + f.c_f[1] * (p - f.p_ref)) * self.gz).reshape(-1)

    def system(self, p, s, pb, old, dt):
        """Residual (2 per block row: oil, water) and the Jacobian's blocks as (rows, cols, values [., 4])."""
        f, g, n = self.f, self.g, self.n
        vdt = g.dx * g.dy * g.dz / dt
        raw = (s - f.swc) / (1.0 - f.swc - f.sor)
        sh = raw.clamp(0.0, 1.0)
        dsh = ((raw >= 0.0) & (raw <= 1.0)).double() / (1.0 - f.swc - f.sor)
        kr = [f.krw_max * sh ** f.nw, f.kro_max * (1.0 - sh) ** f.no]
        dkr = [f.krw_max * f.nw * sh ** (f.nw - 1.0) * dsh, -f.kro_max * f.no * (1.0 - sh) ** (f.no - 1.0) * dsh]
        rho = [f.rho_ref[a] * (1.0 + f.c_f[a] * (p - f.p_ref)) for a in (0, 1)]
        drho = [f.rho_ref[a] * f.c_f[a] for a in (0, 1)]
        mob = [rho[a] * kr[a] / f.mu_ref[a] for a in (0, 1)]
        mob_p = [drho[a] * kr[a] / f.mu_ref[a] for a in (0, 1)]
        mob_s = [rho[a] * dkr[a] / f.mu_ref[a] for a in (0, 1)]
        pot = [p - rho[a] * self.gz for a in (0, 1)]
        pot_p = [1.0 - drho[a] * self.gz for a in (0, 1)]
        por, dpor = self.phi * (1.0 + f.c_r * (p - f.p_ref)), self.phi * f.c_r
        acc = self.accumulation(p, s)
        res = [vdt * (acc[e] - old[e]) for e in (0, 1)]
        sat, dsat = (1.0 - s, s), (-1.0, 1.0)
        diag = []                                              # [e][unknown]
        for e in (0, 1):
            a = 1 - e
            diag.append([vdt * (dpor * rho[a] + por * drho[a]) * sat[e], vdt * dsat[e] * por * rho[a]])
        rows, cols, vals = [], [], []
        for ax in (0, 1, 2):
            m = self.shape[ax] - 1
            if m < 1:
                continue
            lo, hi = (lambda v: v.narrow(ax, 0, m)), (lambda v: v.narrow(ax, 1, m))
            t = self.trans[ax]
            to_lo, to_hi = [None] * 4, [None] * 4              # row lo: column hi; row hi: column lo
            for e in (0, 1):
                a = 1 - e
                d = hi(pot[a]) - lo(pot[a])
                up = lo(pot[a]) >= hi(pot[a])
                zero = torch.zeros_like(d)
                mu = torch.where(up, lo(mob[a]), hi(mob[a]))
                flux = t * mu * d
                l_p = torch.where(up, t * lo(mob_p[a]) * d, zero) - t * mu * lo(pot_p[a])
                l_s = torch.where(up, t * lo(mob_s[a]) * d, zero)
                h_p = torch.where(up, zero, t * hi(mob_p[a]) * d) + t * mu * hi(pot_p[a])
                h_s = torch.where(up, zero, t * hi(mob_s[a]) * d)
                lo(res[e]).sub_(flux)
                hi(res[e]).add_(flux)
                for u, (dl, dh) in enumerate(((l_p, h_p), (l_s, h_s))):
                    lo(diag[e][u]).sub_(dl)
                    hi(diag[e][u]).add_(dh)
                    to_lo[2 * e + u], to_hi[2 * e + u] = -dh, dl
            il, ih = lo(self.idx).reshape(-1), hi(self.idx).reshape(-1)
            rows += [il, ih]
            cols += [ih, il]
            vals += [torch.stack([v.reshape(-1) for v in blk], 1) for blk in (to_lo, to_hi)]
        flat = lambda v: v.reshape(-1)  # noqa: E731
        wres = torch.zeros(self.nw, dtype=torch.float64, device=DEV)
        for k, (w, cells, wi, dz5) in enumerate(self.wells):
            pc = flat(p)[cells]
            pick = lambda v: flat(v)[cells]  # noqa: E731
            q, q_p, q_s, q_b = [], [], [], []
            for a in (0, 1):
                dd = pb[k] - pc + pick(rho[a]) * dz5
                dd_p = -1.0 + drho[a] * dz5
                m, m_p, m_s = pick(mob[a]), pick(mob_p[a]), pick(mob_s[a])
                out = dd <= 0.0 if w.kind == I.PROD else dd < 0.0
                zero = torch.zeros_like(dd)
                vals4 = [wi * m * dd, wi * (m_p * dd + m * dd_p), wi * m_s * dd, wi * m]
                other = [zero] * 4
                if w.kind == I.INJ and a == 0:                 # injection with the total mobility
                    lt = pick(kr[0]) / f.mu_ref[0] + pick(kr[1]) / f.mu_ref[1]
                    lt_s = pick(dkr[0]) / f.mu_ref[0] + pick(dkr[1]) / f.mu_ref[1]
                    r0 = pick(rho[0])
                    other = [wi * r0 * lt * dd, wi * (drho[0] * lt * dd + r0 * lt * dd_p), wi * r0 * lt_s * dd, wi * r0 * lt]
                got = [torch.where(out, x, y) for x, y in zip(vals4, other)]
                for dst, v in zip((q, q_p, q_s, q_b), got):
                    dst.append(v)
            wrow = torch.full_like(cells, n + k)
            for e in (0, 1):
                a = 1 - e
                flat(res[e])[cells] -= q[a]
                flat(diag[e][0])[cells] -= q_p[a]
                flat(diag[e][1])[cells] -= q_s[a]
            zero = torch.zeros_like(pc)
            rows += [cells, wrow]
            cols += [wrow, cells]
            vals.append(torch.stack([-q_b[1], zero, -q_b[0], zero], 1))
            one = torch.ones((), dtype=torch.float64, device=DEV)
            if w.control == I.WRATE:                           # water rate over its target
                sc = (1.0 if w.kind == I.INJ else -1.0) / (f.rho_ref[0] * w.target)
                vals.append(torch.stack([sc * q_p[0], sc * q_s[0], zero, zero], 1))
                wres[k] = sc * q[0].sum() - 1.0
                dw = sc * q_b[0].sum()
            else:
                vals.append(torch.zeros(len(cells), 4, dtype=torch.float64, device=DEV))
                wres[k] = (pb[k] - w.target) / w.target
                dw = one / w.target
            rows.append(wrow[:1])
            cols.append(wrow[:1])
            vals.append(torch.stack([dw, 0 * one, 0 * one, one])[None])
        rows.append(flat(self.idx))
        cols.append(flat(self.idx))
        vals.append(torch.stack([flat(diag[0][0]), flat(diag[0][1]), flat(diag[1][0]), flat(diag[1][1])], 1))
        r = torch.zeros(self.nb, 2, dtype=torch.float64, device=DEV)
        r[:n, 0], r[:n, 1], r[n:, 0] = flat(res[0]), flat(res[1]), wres
        return r, torch.cat(rows), torch.cat(cols), torch.cat(vals)

    def dense(self, rows, cols, vals):
        a = torch.zeros(2 * self.nb, 2 * self.nb, dtype=torch.float64, device=DEV)
        for e in (0, 1):
            for u in (0, 1):
                a[2 * rows + e, 2 * cols + u] = vals[:, 2 * e + u]
        return a

    def step(self, p, s, pb, dt):
        """One time step solved to rounding by Newton with dense solves."""
        old = self.accumulation(p, s)
        n, chop, last = self.n, self.g.sat_chop, math.inf
        for it in range(30):
            r, rows, cols, vals = self.system(p, s, pb, old, dt)
            y = torch.linalg.solve(self.dense(rows, cols, vals), -r.reshape(-1)).reshape(-1, 2)
            ds = y[:n, 1].reshape(self.shape)
            if chop > 0.0:
                ds = ds.clamp(-chop, chop)
            p, s, pb = p + y[:n, 0].reshape(self.shape), (s + ds).clamp(0.0, 1.0), pb + y[n:, 0]
            size = float(y[:n, 1].abs().max())
            if size < 1e-12 or (size < 1e-9 and size >= last):
                return p, s, pb
            last = size
        return None


def _linear_system(geo, seed):
    """A Newton system in mid-run: pressure drawn down around the producers, water banks around the injectors,
    the old level a little behind.  Returns (rowptr, cols, values, b, key)."""
    m = _Model(geo)
    rng = np.random.default_rng(seed + 77)
    t = lambda a: torch.as_tensor(a, dtype=torch.float64, device=DEV)  # noqa: E731
    x, y = torch.arange(geo.nx, device=DEV, dtype=torch.float64), torch.arange(geo.ny, device=DEV, dtype=torch.float64)
    p, s = m.hydrostatic()
    shape = (geo.ny, geo.nx)
    dp, bank = torch.zeros(shape, dtype=torch.float64, device=DEV), torch.zeros(shape, dtype=torch.float64, device=DEV)
    radius = 0.25 * min(geo.nx, geo.ny)
    for w in geo.wells:
        c0 = w.perf_cells[0]
        i, j = c0 % geo.nx, (c0 // geo.nx) % geo.ny
        hump = torch.exp(-((x[None, :] - i) ** 2 + (y[:, None] - j) ** 2) / (radius * rng.uniform(0.5, 1.0)) ** 2)
        dp = dp + (25.0 if w.kind == I.INJ else -25.0) * hump
        if w.kind == I.INJ:
            bank = torch.maximum(bank, hump)
    noise = t(rng.standard_normal(m.shape))
    p = p + dp[None] + 0.05 * noise
    s_old = (0.2 + 0.45 * bank[None] * (0.8 + 0.2 * t(rng.random(m.shape))) * _relative_porosity(m)).clamp(0.2, 0.78)
    s = (s_old + 0.03 * bank[None] * (1.0 - bank[None]) * (1.0 + 0.2 * noise)).clamp(0.2, 0.79)
    old = m.accumulation(p - 0.02 * dp[None], s_old)
    pb = torch.stack([p.reshape(-1)[c[0]] + (12.0 if w.kind == I.INJ else -12.0) for w, c, _, _ in m.wells])
    r, rows, cols, vals = m.system(p, s, pb, old, geo.dt)
    order = torch.argsort(rows * m.nb + cols)
    rows, cols, vals = rows[order], cols[order].to(torch.int32), vals[order].contiguous()
    rp = torch.zeros(m.nb + 1, dtype=torch.int64, device=DEV)
    rp[1:] = torch.cumsum(torch.bincount(rows, minlength=m.nb), 0)
    return rp.to(torch.int32), cols, vals.reshape(-1), (-r).reshape(-1).contiguous(), m.key(p).contiguous()


def _relative_porosity(m):
    """Relative porosity: the water bank runs ahead in the good rock."""
    return m.phi / m.phi.max()


# ------------------------------------------------------- the network -------
_LAYERS = [(0, 8, 32), (0, 32, 32), (1, 32, 32), (1, 32, 32), (2, 32, 32), (2, 32, 32), (3, 32, 32), (3, 32, 32),
           (2, 64, 32), (2, 32, 32), (1, 64, 32), (1, 32, 32), (0, 64, 32), (0, 32, 32), (0, 32, 8)]


def _n_params():
    return sum(27 * ci * co + co for _, ci, co in _LAYERS)


def _network(flat, feat):
    """The U-Net: two 3x3x3 convolutions per level, average pooling, nearest up-sampling, [up, skip], a head."""
    fn = torch.nn.functional
    at, k = 0, 0

    def conv(x, relu=True):
        nonlocal at, k
        _, ci, co = _LAYERS[k]
        w = flat[at:at + 27 * ci * co].reshape(3, 3, 3, co, ci).permute(3, 4, 0, 1, 2)
        b = flat[at + 27 * ci * co:at + 27 * ci * co + co]
        at, k = at + 27 * ci * co + co, k + 1
        y = fn.conv3d(x, w, b, padding=1)
        return torch.relu(y) if relu else y

    x = feat.permute(3, 0, 1, 2)[None]
    skips = []
    for _ in range(3):
        x = conv(conv(x))
        skips.append(x)
        x = fn.avg_pool3d(x, 2, ceil_mode=True, count_include_pad=False)
    x = conv(conv(x))
    for skip in reversed(skips):
        up = x.repeat_interleave(2, 2).repeat_interleave(2, 3).repeat_interleave(2, 4)
        x = torch.cat([up[:, :, :skip.shape[2], :skip.shape[3], :skip.shape[4]], skip], 1)
        x = conv(conv(x))
    return conv(x, relu=False)[0].permute(1, 2, 3, 0)


# ---------------------------------------------------------- 64 bits --------
def exact(case, seed):
    c = case
    if c["kind"] in ("step", "linsys") and c["nx"] * c["ny"] * c["nz"] > 3000:
        return None                                            # dense solves would take too long
    if c["kind"] == "batch" or (c["kind"] in ("train", "predict") and c["nx"] * c["ny"] * c["nz"] > 160000):
        return None
    if c["kind"] == "step":
        m = _Model(_geology(c, seed))
        p, s = m.hydrostatic()
        state = (p, s, m.well_start(p))
        for _ in range(c["warm"] + 1):
            state = m.step(*state, m.g.dt)
            if state is None:
                return None
        return [state[0].reshape(-1), state[1].reshape(-1), state[2]]
    if c["kind"] == "linsys":
        geo = _geology(c, seed)
        rp, ci, val, b, _ = _linear_system(geo, seed)
        m = _Model(geo)
        rows = torch.repeat_interleave(torch.arange(m.nb, device=DEV), (rp[1:] - rp[:-1]).long())
        a = m.dense(rows, ci.long(), val.reshape(-1, 4))
        y = torch.linalg.solve(a, b)
        return y + torch.linalg.solve(a, b - a @ y)
    feat, target = _features(c, seed)
    w = torch.as_tensor(_weights(c, seed), dtype=torch.float64, device=DEV)
    f = torch.as_tensor(feat, dtype=torch.float64, device=DEV)
    if c["kind"] == "predict":
        with torch.no_grad():
            return _network(w, f)
    w.requires_grad_(True)
    t = torch.as_tensor(target, dtype=torch.float64, device=DEV)
    loss = 0.5 * ((_network(w, f)[..., :2] - t) ** 2).sum() / (t.numel() // 2)
    loss.backward()
    g = w.grad
    with torch.no_grad():
        new = w - 1e-4 * g / (g.abs() + 1e-8)
    return dict(loss=float(loss.detach()), grad=g, weights=new)
