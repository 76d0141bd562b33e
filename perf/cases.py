"""Performance cases of the zero-beta MHD library, each through its public entry points.

`listed()` names the cases, `draw(rng)` gives more of the same ranges, `prepare(case, seed)` makes a
user's inputs, grid and parameters on the GPU, `run(state)` is one pass, `work(case)` the bytes and
operations of a pass, and `exact(case, seed)` the outputs in plain 64-bit torch.

The inputs are the seeded synthetic ones of paper_1811_02605_gb300/inputs.py (unit dipole, a 5-mode
perturbation, optionally the flux rope, a 5-mode velocity), evaluated with torch on the device. Steps
start from a saved state that each pass restores, so every pass does the same work. Tolerances are
at the tight end of the range the tests use, so that the outputs are determined by the system that
is solved and not by where an iteration stops.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1811_02605_gb300 as P
from paper_1811_02605_gb300 import autograd as A
from paper_1811_02605_gb300 import inputs as I

DEV = "cuda" if torch.cuda.is_available() else "cpu"
F64 = torch.float64
X0 = 4623.0  # C_w^2 / (1 - C_f)^2 - 1 of the 32x32x64 workload: alpha = X0 / max k~^2 is its SI conditioning
FIELDS = ("br", "bt", "bp", "vr", "vt", "vp")


# ----------------------------------------------------------------------------------------------
# cases
# ----------------------------------------------------------------------------------------------
def _case(name, kind, nr, nt, np_, **kw):
    c = dict(kind=kind, nr=nr, nt=nt, np=np_, r1=20.0, stretch=1.05, rope=False)
    c.update(kw)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # one operator application on the parity grid: the smallest call, bound by launches
        _case("operator_32x32x64", "operator", 32, 32, 64, ncomp=3),
        # whole FP64 steps of the parity workload: small production tests, latency of every iteration counts
        _case("step_fp64_32x32x64", "step", 32, 32, 64, tol=1e-12),
        # a small mixed-precision step at the library's default inner tolerance
        _case("step_mixed_48x48x96", "step", 48, 48, 96, tol=1e-13, precision=1, inner_tol=1e-5, max_outer=60),
        # an ordinary step on a ragged grid (odd nr and nt, np not a multiple of 4) with explicit resistivity
        _case("step_fp64_61x47x118", "step", 61, 47, 118, tol=1e-12, eta=1e-4, r1=10.0, stretch=1.03),
        # FP64 point-Jacobi solve of an SI system that does not fit the L2: the headline iteration
        _case("solve_fp64_160x160x320", "solve", 160, 160, 320, tol=1e-12, r1=30.0, stretch=1.03),
        # mixed-precision SI solve at the size of the flux-rope run: the fast path of that run
        _case("solve_mixed_256x256x512", "solve", 256, 256, 512, tol=1e-13, precision=1, inner_tol=0.1, max_outer=60,
              r1=30.0, stretch=1.02),
        # FP64 steps with PC2 on a middle grid
        _case("step_pc2_96x96x192", "step", 96, 96, 192, tol=1e-12, preconditioner=1, stretch=1.03),
        # the fastest configuration at the size of the flux-rope run: a whole mixed PC2 step
        _case("step_pc2_mixed_256x256x512", "step", 256, 256, 512, tol=1e-13, precision=1, inner_tol=1e-3,
              max_outer=60, preconditioner=1, r1=30.0, stretch=1.02, rope=True),
        # independent systems of uneven size in one launch (the batched workload's sizes)
        _case("batch_8_of_32_to_96", "batch", 96, 96, 192, count=8, tol=1e-12),
        # reverse-mode gradient of two steps (forward, recomputation and adjoint)
        _case("gradient_48x48x96", "gradient", 48, 48, 96, nsteps=2, tol=1e-12, stretch=1.05 ** 0.5),
        # super time-stepping viscosity and implicit resistivity, PC2 in the SI solves
        _case("step_sts_resistive_64x64x128", "step", 64, 64, 128, tol=1e-13, viscosity_sts=1, preconditioner=1,
              resistivity_implicit=1, eta=1e-3),
        # coefficients, force, induction and diagnostics at the size of the flux-rope run, no solve
        _case("explicit_256x256x512", "explicit", 256, 256, 512, eta=1e-4, r1=30.0, stretch=1.02, rope=True),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """Kinds, options and sizes spread over the ranges that the listed cases stand for."""
    kind = rng.choice(["operator", "step", "step", "step", "solve", "solve", "batch", "gradient", "explicit"])
    hi = {"operator": 256, "step": 112, "solve": 176, "batch": 96, "gradient": 56, "explicit": 256}[kind]
    lo = {"operator": 6, "step": 16, "solve": 16, "batch": 24, "gradient": 12, "explicit": 12}[kind]
    nt = _log_int(rng, lo, hi)
    nr = max(4, int(round(nt * rng.uniform(0.8, 1.2))))
    np_ = max(8, 2 * int(round(nt * rng.uniform(0.9, 1.1))))
    if rng.random() < 0.5:
        np_ = -(-np_ // 32) * 32
    c = _case(None, kind, nr, nt, np_, r1=rng.choice([10.0, 20.0, 30.0]), stretch=round(1.0 + rng.uniform(0.5, 1.6) / nr, 4))
    if kind == "operator":
        c["ncomp"] = rng.choice([1, 2, 3])
    elif kind == "batch":
        c.update(count=rng.randint(3, 10), tol=1e-12)
    elif kind == "gradient":
        c.update(nsteps=rng.choice([1, 2, 3]), tol=1e-12)
    elif kind == "explicit":
        c["eta"] = rng.choice([0.0, 1e-4])
    else:
        o = rng.choice([dict(tol=1e-12), dict(tol=1e-12), dict(tol=1e-12, pcg_variant=1), dict(tol=1e-12, preconditioner=1),
                        dict(tol=1e-13, precision=1, inner_tol=0.1, max_outer=60),
                        dict(tol=1e-13, precision=1, inner_tol=1e-5, mixed_restart=1, max_outer=60),
                        dict(tol=1e-13, precision=1, inner_tol=1e-3, preconditioner=1, max_outer=60)])
        c.update(o)
        if kind == "step" and rng.random() < 0.25:
            c.update(viscosity_sts=1)
        if kind == "step" and rng.random() < 0.25:
            c.update(resistivity_implicit=1, eta=1e-3)
    return c


def work(case):
    """Bytes that a pass cannot do without (an iterative solve sweeps its vectors once per iteration: x, r and p read and
    written) and its operations, with nominal iteration counts."""
    N = case["nr"] * case["nt"] * case["np"]
    k = case["kind"]
    if k == "operator":
        return dict(bytes=16.0 * case["ncomp"] * N, flops=13.0 * case["ncomp"] * N)
    if k == "explicit":
        return dict(bytes=8.0 * N * (6 + 6 + 3 + 9 + 6), flops=330.0 * N)
    if k == "batch":
        return dict(bytes=sum(_solve_work(dict(case, nt=d.nt), d.nr * d.nt * d.np)[0] for d in _batch_descs(case)),
                    flops=sum(_solve_work(dict(case, nt=d.nt), d.nr * d.nt * d.np)[1] for d in _batch_descs(case)))
    b, f = _solve_work(case, N)
    if k == "solve":
        return dict(bytes=b, flops=f)
    b, f = 2.1 * b + 12 * 8 * N, 2.1 * f + 330.0 * N
    if k == "gradient":
        b, f = 2.5 * case["nsteps"] * b, 2.5 * case["nsteps"] * f
    return dict(bytes=b, flops=f)


def _solve_work(case, N):
    pc2 = case.get("preconditioner", 0) == 1
    its = (45.0 * (case["nt"] / 32.0) ** 0.4 if pc2 else 235.0 * (case["nt"] / 32.0) ** 0.8) * -math.log10(case["tol"]) / 9.0
    word = 4 if case.get("precision", 0) == 1 else 8
    return its * (8 if pc2 else 6) * 3 * word * N, its * (69.0 + (30.0 if pc2 else 0.0)) * N


# ----------------------------------------------------------------------------------------------
# inputs
# ----------------------------------------------------------------------------------------------
def _desc(c):
    return I.GridDesc(c["nr"], c["nt"], c["np"], 1.0, c["r1"], c["stretch"])


def _batch_descs(c):
    """Grids of a batch: nt spread from 32 (or less) to the case's own, nr = nt, np = 2 nt, stretch in [1.02, 1.08]."""
    lo = min(32, c["nt"])
    out = []
    for s in range(c["count"]):
        nt = int(round(lo + (c["nt"] - lo) * s / max(1, c["count"] - 1)))
        out.append(I.GridDesc(nt, nt, 2 * nt, 1.0, 20.0, 1.02 + 0.06 * ((5 * s) % 8) / 7.0))
    return out


def _t(a):
    return torch.as_tensor(np.asarray(a, dtype=np.float64), device=DEV)


def _modes(m, x, y, z, tx, ty, tz):
    """Component along (tx, ty, tz) of the smooth mode field at Cartesian points (x, y, z)."""
    out = 0.0
    for k, u, p in zip(m.k, m.u, m.phase):
        s = torch.sin(float(k[0]) * x + float(k[1]) * y + float(k[2]) * z + float(p))
        out = out + m.amp * s * (float(u[0]) * tx + float(u[1]) * ty + float(u[2]) * tz)
    return out


def _rope(rp, x, y, z, tx, ty, tz):
    """Component along (tx, ty, tz) of the twisted rope's vector potential (axis circle around the x axis)."""
    n = [float(v) for v in rp.normal]
    d0 = [q - float(c) for q, c in zip((x, y, z), rp.centre)]
    yn = n[0] * d0[0] + n[1] * d0[1] + n[2] * d0[2]
    yp = [q - m * yn for q, m in zip(d0, n)]
    pl = torch.sqrt(yp[0] ** 2 + yp[1] ** 2 + yp[2] ** 2).clamp_min(1e-12)
    e = [q / pl for q in yp]
    dv = [q - rp.R * w for q, w in zip(d0, e)]
    d = torch.sqrt(dv[0] ** 2 + dv[1] ** 2 + dv[2] ** 2)
    cross = lambda a, b: [a[1] * b[2] - a[2] * b[1], a[2] * b[0] - a[0] * b[2], a[0] * b[1] - a[1] * b[0]]  # noqa: E731
    t = cross(n, e)
    psi = cross(t, [q / d.clamp_min(1e-14) for q in dv])
    g = torch.where((pl > 1e-12) & (d < 6.0 * rp.a), torch.exp(-d * d / (rp.a * rp.a)), torch.zeros_like(d))
    a_psi, a_ax = rp.B0 * 0.5 * d * g, rp.tau * rp.B0 * 0.5 * rp.a * rp.a * g
    return sum((a_psi * p + a_ax * q) * w for p, q, w in zip(psi, t, (tx, ty, tz)))


class _Angles:
    def __init__(self, d):
        th, s, c = I.theta_nodes(d.nt)
        self.r = _t(I.radial_nodes(d))
        self.rc = 0.5 * (self.r[1:] + self.r[:-1])
        self.sn, self.cn = _t(s), _t(c)
        self.dth, self.dph = math.pi / d.nt, 2.0 * math.pi / d.np
        thc = (torch.arange(d.nt, device=DEV, dtype=F64) + 0.5) * self.dth
        self.sc, self.cc = torch.sin(thc), torch.cos(thc)
        phn = torch.arange(d.np, device=DEV, dtype=F64) * self.dph
        self.phn, self.phc = phn, phn + 0.5 * self.dph


def _field_b(d, modes, rope):
    """Face-averaged B of dipole + modes (+ rope): circulation of the vector potential around each face over its area."""
    g = _Angles(d)
    c3 = lambda a: a[:, None, None]  # noqa: E731
    c2 = lambda a: a[None, :, None]  # noqa: E731

    def integral(r, st, ct, ph, along, length, dip):
        sp, cp = torch.sin(ph)[None, None], torch.cos(ph)[None, None]
        tang = {"r": (st * cp, st * sp, ct + 0 * sp), "t": (ct * cp, ct * sp, -st + 0 * sp),
                "p": (-sp + 0 * st, cp + 0 * st, 0 * sp + 0 * st)}[along]
        pos = (r * st * cp, r * st * sp, r * ct + 0 * sp)
        a = _modes(modes, *pos, *tang)
        if rope:
            a = a + _rope(I.default_rope(), *pos, *tang)
        return (a + dip) * length

    rm = 0.5 * (g.r[1:] + g.r[:-1])
    Lr = integral(c3(rm), c2(g.sn), c2(g.cn), g.phn, "r", c3(g.r[1:] - g.r[:-1]), 0.0)
    Lt = integral(c3(g.r), c2(g.sc), c2(g.cc), g.phn, "t", c3(g.r * g.dth), 0.0)
    Lp = integral(c3(g.r), c2(g.sn), c2(g.cn), g.phc, "p", c3(g.r) * c2(g.sn) * g.dph, c2(g.sn) / c3(g.r) ** 2)
    br = (Lt - torch.roll(Lt, -1, 2) + Lp[:, 1:] - Lp[:, :-1]) / (c3(g.r ** 2) * c2(g.cn[:-1] - g.cn[1:]) * g.dph)
    ring = 0.5 * (g.r[1:] ** 2 - g.r[:-1] ** 2)
    bt = torch.zeros((d.nr, d.nt + 1, d.np), device=DEV, dtype=F64)
    ft = Lp[:-1] - Lp[1:] + torch.roll(Lr, -1, 2) - Lr
    bt[:, 1:-1] = ft[:, 1:-1] / (c3(ring) * c2(g.sn[1:-1]) * g.dph)
    bp = (Lr[:, :-1] - Lr[:, 1:] + Lt[1:] - Lt[:-1]) / (c3(ring) * g.dth)
    return br.contiguous(), bt, bp.contiguous()


def _field_v(d, modes, ramp):
    """Smooth mode field at the cell centres on the spherical basis, [3, nr, nt, np]."""
    g = _Angles(d)
    r, st, ct = g.rc[:, None, None], g.sc[None, :, None], g.cc[None, :, None]
    sp, cp = torch.sin(g.phc)[None, None], torch.cos(g.phc)[None, None]
    pos = (r * st * cp, r * st * sp, r * ct + 0 * sp)
    w = (1.0 - torch.exp(-(r - d.r0) / ramp)) if ramp else 1.0
    basis = ((st * cp, st * sp, ct + 0 * sp), (ct * cp, ct * sp, -st + 0 * sp), (-sp + 0 * st, cp + 0 * st, 0 * sp + 0 * st))
    return torch.stack([_modes(modes, *pos, *b) * w for b in basis])


def _state(d, seed, rope):
    rng = np.random.default_rng(seed)
    bm, vm = I.draw_modes(rng, 1e-3, 1.0 / d.r1), I.draw_modes(rng, 1e-2, 1.0 / d.r1)
    br, bt, bp = _field_b(d, bm, rope)
    v = _field_v(d, vm, 0.1)
    return dict(br=br, bt=bt, bp=bp, vr=v[0].clone(), vt=v[1].clone(), vp=v[2].clone())


def _volume_density(d):
    g = _Angles(d)
    return ((d.r0 / g.rc) ** 2 * (g.r[1:] ** 3 - g.r[:-1] ** 3) / 3.0)[:, None] * (g.cn[:-1] - g.cn[1:])[None] * g.dph


def _max_kt2(d):
    g = _Angles(d)
    k = 1.0 / (g.r[1:] - g.r[:-1])[:, None] ** 2 + 1.0 / (g.rc * g.dth)[:, None] ** 2 + 1.0 / (g.rc[:, None] * g.sc[None] * g.dph) ** 2
    return float(k.max())


def _rhs(d, seed, ncomp=3):
    """rho V times a smooth field: the right-hand side of an implicit system."""
    m = I.draw_modes(np.random.default_rng(seed), 1.0, 1.0 / d.r1)
    return (_field_v(d, m, 0.0)[:ncomp] * _volume_density(d)[None, :, :, None]).contiguous()


_PARAMS = ("tol", "precision", "inner_tol", "max_outer", "mixed_restart", "viscosity_sts", "pcg_variant",
           "resistivity_implicit", "preconditioner", "eta")


def _param_kw(c):
    return dict({k: c[k] for k in _PARAMS if k in c}, nu=1e-3, cfl=0.4)


def _features(c):
    f = P.RESERVE_PC2 if c.get("preconditioner") else P.RESERVE_CG if c.get("pcg_variant") else 0 if c.get("precision") else P.RESERVE_PC1
    f |= P.RESERVE_MIXED if c.get("precision") else 0
    return f | (P.RESERVE_RESISTIVITY if c.get("resistivity_implicit") else 0)


def _grid(d):
    return P.mhd_grid_create(d.nr, d.nt, d.np, d.r0, d.r1, d.stretch)


def _fields(s):
    return P.make_fields(*(s[k] for k in FIELDS))


def prepare(case, seed):
    d, kind = _desc(case), case["kind"]
    s = dict(kind=kind)
    if kind == "batch":
        descs = _batch_descs(case)
        s.update(grids=[_grid(q) for q in descs], alphas=[X0 / _max_kt2(q) for q in descs],
                 b=[_rhs(q, 1000 * seed + n) for n, q in enumerate(descs)], params=P.make_params(tol=case["tol"]))
        s["x"] = [torch.zeros_like(b) for b in s["b"]]
        P.pcg_batch_reserve(s["grids"], s["alphas"], s["b"], s["x"], s["params"])
        return s
    g = s["grid"] = _grid(d)
    if kind == "operator":
        s.update(alpha=X0 / _max_kt2(d), p=_field_v(d, I.draw_modes(np.random.default_rng(seed), 1.0, 1.0 / d.r1), 0.0)[:case["ncomp"]].contiguous())
        s["q"] = torch.empty_like(s["p"])
    elif kind == "solve":
        s.update(alpha=X0 / _max_kt2(d), b=_rhs(d, seed), params=P.make_params(**_param_kw(case)))
        s["x"] = torch.zeros_like(s["b"])
        P.mhd_grid_reserve(g, _features(case))
    elif kind == "gradient":
        s.update(saved=_state(d, seed, case["rope"]), nsteps=case["nsteps"], kw=_param_kw(case), target=_t(I.outer_target(d, seed)))
        P.mhd_grid_reserve(g, P.RESERVE_PC1 | P.RESERVE_ADJOINT)
    else:
        s["saved"] = _state(d, seed, case["rope"])
        s["now"] = {k: torch.empty_like(v) for k, v in s["saved"].items()}
        s["fields"] = _fields(s["now"])
        s["params"] = P.make_params(**_param_kw(case))
        if kind == "step":
            P.mhd_grid_reserve(g, _features(case))
        else:
            s.update(eta=case["eta"], b=torch.empty((3, d.nr, d.nt, d.np), device=DEV, dtype=F64),
                     vbar=torch.stack([s["saved"][k] for k in ("vr", "vt", "vp")]))
    return s


def run(s):
    kind = s["kind"]
    if kind == "operator":
        P.mhd_apply_operator(s["grid"], s["alpha"], s["p"], s["q"])
        return s["q"]
    if kind == "solve":
        s["x"].zero_()
        status = P.pcg_solve(s["grid"], s["alpha"], s["b"], s["x"], s["params"])[0]
        return _checked(status, s["x"])
    if kind == "batch":
        torch._foreach_zero_(s["x"])
        status = P.pcg_solve_batched(s["grids"], s["alphas"], s["b"], s["x"], s["params"])[0]
        return _checked(status, s["x"])
    if kind == "gradient":
        start = {k: v.detach().requires_grad_(True) for k, v in s["saved"].items()}
        out = A.simulate(s["grid"], start, s["nsteps"], **s["kw"])
        loss = 0.5 * ((out["br"][-1] - s["target"]) ** 2).sum()
        loss.backward()
        return dict(loss=loss.detach(), out={k: out[k].detach() for k in FIELDS}, grad={k: start[k].grad for k in FIELDS})
    torch._foreach_copy_([s["now"][k] for k in FIELDS], [s["saved"][k] for k in FIELDS])
    if kind == "step":
        status, info = P.mhd_step(s["grid"], s["params"], s["fields"])
        return _checked(status, dict(s["now"], dt=info["dt"], alpha_si=info["alpha_si"]))
    co = P.mhd_step_coeffs(s["grid"], s["params"], s["fields"])
    P.mhd_force(s["grid"], s["fields"], co["dt"], s["b"])
    P.mhd_induction(s["grid"], s["vbar"], s["eta"], co["dt"], s["fields"])
    di = P.mhd_diagnostics(s["grid"], s["fields"])  # its max |div B| is rounding noise and is not returned
    return dict(s["now"], b=s["b"], **{k: co[k] for k in ("dt", "cf", "cw", "alpha_si", "alpha_nu")},
                **{k: di[k] for k in ("magnetic_energy", "kinetic_energy", "int_jxb", "int_jdotb")})


def _checked(status, out):
    if status != P.MHD_OK:
        raise RuntimeError(f"status {P.STATUS_NAMES[status]}")
    return out


# ----------------------------------------------------------------------------------------------
# the same results in plain 64-bit torch
# ----------------------------------------------------------------------------------------------
class _Exact:
    """Geometry, implicit solves and explicit updates of one grid, as whole-array torch expressions."""

    def __init__(self, d):
        self.d, g = d, _Angles(d)
        self.__dict__.update(g.__dict__)
        self.ring = 0.5 * (g.r[1:] ** 2 - g.r[:-1] ** 2)
        self.band = g.cn[:-1] - g.cn[1:]
        self.rho = (d.r0 / g.rc) ** 2
        self.vol = ((g.r[1:] ** 3 - g.r[:-1] ** 3) / 3.0)[:, None] * self.band[None] * g.dph
        self.rhoV = (self.rho[:, None] * self.vol)[None, :, :, None]
        # M = a_i band_j + alpha (radial differences x band_j + Q_i (theta differences + phi differences P_j))
        self.a = self.rho * (g.r[1:] ** 3 - g.r[:-1] ** 3) / 3.0 * g.dph
        gap = torch.cat([(g.rc[:1] - g.r[:1]), g.rc[1:] - g.rc[:-1]])
        self.R = torch.cat([(d.r0 / g.r[:-1]) ** 2 * g.r[:-1] ** 2 * g.dph / gap, torch.zeros(1, device=DEV, dtype=F64)])
        self.Q = self.rho * self.ring * g.dph / (g.rc * g.dth)
        self.Pj = (g.dth / g.dph) ** 2 / g.sc
        self.lo = torch.cat([2.0 * d.r0 - g.rc[:1], g.rc])      # radii on either side of a shell of nodes
        self.hi = torch.cat([g.rc, 2.0 * g.r[-1:] - g.rc[-1:]])
        self.kt2 = (1.0 / (g.r[1:] - g.r[:-1])[:, None] ** 2 + 1.0 / (g.rc * g.dth)[:, None] ** 2 +
                    1.0 / (g.rc[:, None] * g.sc[None] * g.dph) ** 2)
        self.modes = None

    # -- the implicit operator and its direct solve (Fourier in phi, eigenvectors in theta, tridiagonal in r)
    def apply_K(self, u):
        z = torch.zeros_like
        dr = torch.cat([u[:, :1], u[:, 1:] - u[:, :-1], z(u[:, :1])], 1) * (self.R[:, None] * self.band[None])[None, :, :, None]
        dt = torch.cat([z(u[:, :, :1]), u[:, :, 1:] - u[:, :, :-1], z(u[:, :, :1])], 2) * self.sn[None, None, :, None]
        ph = (2.0 * u - torch.roll(u, 1, 3) - torch.roll(u, -1, 3)) * self.Pj[None, None, :, None]
        return dr[:, :-1] - dr[:, 1:] + self.Q[None, :, None, None] * (dt[:, :, :-1] - dt[:, :, 1:] + ph)

    def apply_M(self, alpha, u):
        return self.rhoV * u + alpha * self.apply_K(u)

    def _direct(self, alpha, b):
        d, nm = self.d, self.d.np // 2 + 1
        if self.modes is None:
            m = torch.arange(nm, device=DEV, dtype=F64)
            lam = 2.0 - 2.0 * torch.cos(2.0 * math.pi * m / d.np)
            T = torch.diag(self.sn[:-1] + self.sn[1:]) - torch.diag(self.sn[1:-1], 1) - torch.diag(self.sn[1:-1], -1)
            S = (T[None] + torch.diag_embed(lam[:, None] * self.Pj[None])) / torch.sqrt(self.band[:, None] * self.band[None])
            self.modes = torch.linalg.eigh(S)
        mu, U = self.modes
        sb = torch.sqrt(self.band)[None, None, :, None]
        c = b.shape[0]
        X = torch.view_as_real(torch.fft.rfft(b / sb, dim=3)).permute(3, 2, 0, 1, 4).reshape(nm, d.nt, -1)
        Y = (U.transpose(1, 2) @ X).reshape(nm, d.nt, c, d.nr, 2)
        e = alpha * mu[:, :, None, None]
        off = -alpha * self.R
        piv, ys = [], []
        for i in range(d.nr):
            dia = self.a[i] + alpha * (self.R[i] + self.R[i + 1]) + e * self.Q[i]
            y = Y[:, :, :, i]
            if i:
                w = off[i] / piv[-1]
                dia, y = dia - w * off[i], y - w * ys[-1]
            piv.append(dia)
            ys.append(y)
        out = [ys[-1] / piv[-1]]
        for i in range(d.nr - 2, -1, -1):
            out.append((ys[i] - off[i + 1] * out[-1]) / piv[i])
        X = (U @ torch.stack(out[::-1], 3).reshape(nm, d.nt, -1)).reshape(nm, d.nt, c, d.nr, 2).permute(2, 3, 1, 0, 4)
        return torch.fft.irfft(torch.view_as_complex(X.contiguous()), n=d.np, dim=3) / sb

    def solve(self, alpha, b):
        x = self._direct(alpha, b)
        return x + self._direct(alpha, b - self.apply_M(alpha, x))

    # -- explicit parts
    def centre_b(self, br, bt, bp):
        ph = self.phc
        def pole(face):
            h = (face * torch.cos(ph)).sum(-1, keepdim=True) * torch.cos(ph) + (face * torch.sin(ph)).sum(-1, keepdim=True) * torch.sin(ph)
            return 0.5 * (face + h * 2.0 / (self.d.np * math.cos(self.dth)))
        t = torch.cat([pole(bt[:, 1:2]), 0.5 * (bt[:, 1:-2] + bt[:, 2:-1]), pole(bt[:, -2:-1])], 1)
        return torch.stack([0.5 * (br[:-1] + br[1:]), t, 0.5 * (bp + torch.roll(bp, -1, 2))])

    def current(self, br, bt, bp, walls=True):
        """Edge currents (radial, theta, phi edges); walls False: none on the tangential edges of r0 and r1."""
        rc, sc, cc, dth, dph = self.rc[:, None, None], self.sc[None, :, None], self.cc[None, :, None], self.dth, self.dph
        km = lambda a: torch.roll(a, 1, 2)  # noqa: E731
        area = rc ** 2 * (cc[:, :-1] - cc[:, 1:]) * dph
        jr = (rc * sc[:, 1:] * dph * bp[:, 1:] - rc * sc[:, :-1] * dph * bp[:, :-1] - rc * dth * (bt - km(bt))[:, 1:-1]) / area
        n = bp[:, :1].sum(2, keepdim=True) * sc[:, :1] * dph / (rc * (1.0 - cc[:, :1]) * 2.0 * math.pi)
        s = -bp[:, -1:].sum(2, keepdim=True) * sc[:, -1:] * dph / (rc * (1.0 + cc[:, -1:]) * 2.0 * math.pi)
        jr = torch.cat([n.expand(-1, -1, self.d.np), jr, s.expand(-1, -1, self.d.np)], 1)
        lo, hi = self.lo[:, None, None], self.hi[:, None, None]
        two = 0.5 * (hi ** 2 - lo ** 2)
        pl, ph = torch.cat([bp[:1], bp]), torch.cat([bp, bp[-1:]])
        tl, th = torch.cat([bt[:1], bt]), torch.cat([bt, bt[-1:]])
        jt = (lo * sc * dph * pl + (hi - lo) * (br - km(br)) - hi * sc * dph * ph) / (sc * two * dph)
        jp = ((hi - lo) * (br[:, :-1] - br[:, 1:]) + hi * dth * th[:, 1:-1] - lo * dth * tl[:, 1:-1]) / (two * dth)
        if not walls:
            jt = torch.cat([torch.zeros_like(jt[:1]), jt[1:-1], torch.zeros_like(jt[:1])])
            jp = torch.cat([torch.zeros_like(jp[:1]), jp[1:-1], torch.zeros_like(jp[:1])])
        z = torch.zeros_like(jp[:, :1])
        return jr, jt, torch.cat([z, jp, z], 1)

    def centre_j(self, jr, jt, jp):
        kp = lambda a: a + torch.roll(a, -1, 2)  # noqa: E731
        p = jp[:-1] + jp[1:]
        p = torch.cat([0.5 * p[:, 1:2], 0.25 * (p[:, 1:-2] + p[:, 2:-1]), 0.5 * p[:, -2:-1]], 1)
        return torch.stack([0.25 * kp(jr[:, :-1] + jr[:, 1:]), 0.25 * kp(jt[:-1] + jt[1:]), p])

    def force(self, v, br, bt, bp, dt):
        """rho V dt F(v, B), first-order upwind by the sign of the cell's own velocity."""
        gap = self.rc[1:] - self.rc[:-1]
        ilo = torch.cat([0.5 / (self.rc[:1] - self.d.r0), 1.0 / gap])[None, :, None, None]
        ihi = torch.cat([1.0 / gap, torch.zeros(1, device=DEV, dtype=F64)])[None, :, None, None]
        up = lambda k, back, ahead: torch.where(v[k][None] > 0.0, back, ahead)  # noqa: E731
        z = torch.zeros_like
        dr = up(0, (v - torch.cat([-v[:, :1], v[:, :-1]], 1)) * ilo, (torch.cat([v[:, 1:], v[:, -1:]], 1) - v) * ihi)
        iht = (1.0 / (self.rc * self.dth))[None, :, None, None]
        dn = (v[:, :, 1:] - v[:, :, :-1]) * iht
        dt_ = up(1, torch.cat([z(v[:, :, :1]), dn], 2), torch.cat([dn, z(v[:, :, :1])], 2))
        ihp = (1.0 / (self.rc[:, None] * self.sc[None] * self.dph))[None, :, :, None]
        dp = up(2, (v - torch.roll(v, 1, 3)) * ihp, (torch.roll(v, -1, 3) - v) * ihp)
        adv = v[0][None] * dr + v[1][None] * dt_ + v[2][None] * dp
        irc, cot = 1.0 / self.rc[:, None, None], (self.cc / self.sc)[None, :, None]
        adv = adv + torch.stack([-(v[1] ** 2 + v[2] ** 2) * irc, (v[0] * v[1] - v[2] ** 2 * cot) * irc,
                                 (v[0] * v[2] + v[1] * v[2] * cot) * irc])
        B, J = self.centre_b(br, bt, bp), self.centre_j(*self.current(br, bt, bp))
        return self.rhoV * dt * (-adv + torch.linalg.cross(J, B, dim=0) / self.rho[None, :, None, None])

    def ct(self, er, et, ep, dt, br, bt, bp):
        """B - dt curl E on the faces."""
        r, sn, dth, dph = self.r[:, None, None], self.sn[None, :, None], self.dth, self.dph
        kp = lambda a: torch.roll(a, -1, 2)  # noqa: E731
        lp = r * sn * dph * ep
        cr = (r * dth * (et - kp(et)) + lp[:, 1:] - lp[:, :-1]) / (r ** 2 * self.band[None, :, None] * dph)
        lr = (r[1:] - r[:-1]) * er
        ring = self.ring[:, None, None]
        c = (lp[:-1] - lp[1:] + kp(lr) - lr)[:, 1:-1] / (ring * sn[:, 1:-1] * dph)
        ctt = torch.cat([torch.zeros_like(bt[:, :1]), c, torch.zeros_like(bt[:, :1])], 1)
        lt = r * dth * et
        cp = (lr[:, :-1] - lr[:, 1:] + lt[1:] - lt[:-1]) / (ring * dth)
        return br - dt * cr, bt - dt * ctt, bp - dt * cp

    def induction(self, v, eta, dt, br, bt, bp):
        E = -torch.linalg.cross(v, self.centre_b(br, bt, bp), dim=0)
        if eta:
            E = E + eta * self.centre_j(*self.current(br, bt, bp))
        km = lambda a: a + torch.roll(a, 1, 2)  # noqa: E731
        mean = lambda a: a.mean(2, keepdim=True).expand(-1, -1, self.d.np)  # noqa: E731
        er = torch.cat([mean(E[0][:, :1]), 0.25 * km(E[0][:, :-1] + E[0][:, 1:]), mean(E[0][:, -1:])], 1)
        et = torch.cat([torch.zeros_like(E[1][:1]), 0.25 * km(E[1][:-1] + E[1][1:]), 0.5 * km(E[1][-1:])])
        p = E[2][:, :-1] + E[2][:, 1:]
        p = torch.cat([torch.zeros_like(p[:1]), 0.25 * (p[:-1] + p[1:]), 0.5 * p[-1:]])
        z = torch.zeros_like(p[:, :1])
        return self.ct(er, et, torch.cat([z, p, z], 1), dt, br, bt, bp)

    def resist(self, dte, br, bt, bp):
        """The faces after B + dte curl J(B) = B*: CG in the inner product that makes curl J self-adjoint."""
        r, sn, dth, dph = self.r[:, None, None], self.sn[None, :, None], self.dth, self.dph
        rc = self.rc[:, None, None]
        gap = torch.cat([self.rc[:1] - self.r[:1], self.rc[1:] - self.rc[:-1], self.r[-1:] - self.rc[-1:]])[:, None, None]
        W = (r ** 2 * self.band[None, :, None] * dph * gap, self.ring[:, None, None] * sn * dph * rc * dth,
             self.ring[:, None, None] * dth * rc * self.sc[None, :, None] * dph)
        dot = lambda a, b: sum(float((w * p * q).sum()) for w, p, q in zip(W, a, b))  # noqa: E731
        op = lambda f: self.ct(*self.current(*f, walls=False), -dte, *f)  # noqa: E731
        x = [br, bt, bp]
        q = op(x)
        res = [b - m for b, m in zip((br, bt, bp), q)]
        p, rho, stop = res, dot(res, res), 1e-30 * dot(x, x)
        for _ in range(5000):
            if rho <= stop:
                break
            q = op(p)
            al = rho / dot(p, q)
            x = [a + al * b for a, b in zip(x, p)]
            res = [a - al * b for a, b in zip(res, q)]
            new = dot(res, res)
            p, rho = [a + new / rho * b for a, b in zip(res, p)], new
        return self.ct(*self.current(*x, walls=False), dte, br, bt, bp)

    def sts(self, nu, dt, y0):
        """RKL2 stages of dv/dt = -nu (rho V)^-1 K v."""
        s2 = (self.R[:-1] + self.R[1:])[:, None] * self.band[None] + self.Q[:, None] * (self.sn[:-1] + self.sn[1:] + 2.0 * self.Pj)[None]
        off = s2.clone()
        off[0] -= self.R[0] * self.band
        lam = nu * float(((s2 + off) / self.rhoV[0, :, :, 0]).max())
        s = 2
        while (s * s + s - 2) / 2.0 < dt * lam:
            s += 1
        L = lambda u: -nu * dt * self.apply_K(u) / self.rhoV  # noqa: E731
        b = lambda j: 1.0 / 3.0 if j < 2 else (j * j + j - 2) / (2.0 * j * (j + 1))  # noqa: E731
        w1, l0 = 4.0 / (s * s + s - 2), L(y0)
        y1, y2 = y0 + b(1) * w1 * l0, y0
        for j in range(2, s + 1):
            mu, nv = (2.0 * j - 1.0) / j * b(j) / b(j - 1), -(j - 1.0) / j * b(j) / b(j - 2)
            y1, y2 = mu * y1 + nv * y2 + (1.0 - mu - nv) * y0 + mu * w1 * L(y1) - (1.0 - b(j - 1)) * mu * w1 * l0, y1
        return y1

    def coeffs(self, f, nu=1e-3, cfl=0.4):
        v = torch.stack([f["vr"], f["vt"], f["vp"]])
        B = self.centre_b(f["br"], f["bt"], f["bp"])
        kv = math.sqrt(float((self.kt2[:, :, None] * (v * v).sum(0)).max()))
        ka = math.sqrt(float((self.kt2[:, :, None] * (B * B).sum(0) / self.rho[:, None, None]).max()))
        dt = cfl / kv
        cf, cw = dt * kv, dt * ka
        return dict(dt=dt, cf=cf, cw=cw, alpha_si=max(cw * cw / (1.0 - cf) ** 2 - 1.0, 0.0) / float(self.kt2.max()), alpha_nu=nu * dt)

    def step(self, f, c, nu=1e-3):
        co = self.coeffs({k: t.detach() for k, t in f.items()}, nu)
        dt, a = co["dt"], co["alpha_si"]
        eta, implicit = c.get("eta", 0.0), c.get("resistivity_implicit", 0)
        v, B = torch.stack([f["vr"], f["vt"], f["vp"]]), (f["br"], f["bt"], f["bp"])
        b0 = self.force(v, *B, dt)
        dp = _Solve.apply(b0, self, a)
        B = self.induction(v + 0.5 * dp, 0.0 if implicit else eta, dt, *B)
        if implicit:
            B = self.resist(dt * eta, *B)
        dc = _Solve.apply(0.5 * (b0 + self.force(v + dp, *B, dt)), self, a)
        v = v + dc
        v = self.sts(nu, dt, v) if c.get("viscosity_sts") else _Solve.apply(self.rhoV * v, self, co["alpha_nu"])
        return dict(br=B[0], bt=B[1], bp=B[2], vr=v[0], vt=v[1], vp=v[2]), co

    def diagnostics(self, f):
        v, B = torch.stack([f["vr"], f["vt"], f["vp"]]), self.centre_b(f["br"], f["bt"], f["bp"])
        J, V = self.centre_j(*self.current(f["br"], f["bt"], f["bp"])), self.vol[:, :, None]
        return dict(magnetic_energy=float((0.5 * (B * B).sum(0) * V).sum()),
                    kinetic_energy=float((0.5 * self.rho[:, None, None] * (v * v).sum(0) * V).sum()),
                    int_jxb=float((torch.linalg.cross(J, B, dim=0).square().sum(0).sqrt() * V).sum()),
                    int_jdotb=float(((J * B).sum(0).abs() * V).sum()))


class _Solve(torch.autograd.Function):
    """x = M_alpha^-1 b with the symmetric M_alpha held fixed."""

    @staticmethod
    def forward(ctx, b, ex, alpha):
        ctx.ex, ctx.alpha = ex, alpha
        return ex.solve(alpha, b)

    @staticmethod
    def backward(ctx, g):
        return ctx.ex.solve(ctx.alpha, g), None, None


def exact(case, seed):
    d, kind = _desc(case), case["kind"]
    if kind == "batch":
        return [_Exact(q).solve(X0 / _max_kt2(q), _rhs(q, 1000 * seed + n)) for n, q in enumerate(_batch_descs(case))]
    ex = _Exact(d)
    if kind == "operator":
        m = I.draw_modes(np.random.default_rng(seed), 1.0, 1.0 / d.r1)
        return ex.apply_M(X0 / _max_kt2(d), _field_v(d, m, 0.0)[:case["ncomp"]])
    if kind == "solve":
        return ex.solve(X0 / _max_kt2(d), _rhs(d, seed))
    f = _state(d, seed, case["rope"])
    if kind == "gradient":
        start = {k: t.requires_grad_(True) for k, t in f.items()}
        now = start
        for _ in range(case["nsteps"]):
            now = ex.step(now, case)[0]
        loss = 0.5 * ((now["br"][-1] - _t(I.outer_target(d, seed))) ** 2).sum()
        loss.backward()
        return dict(loss=loss.detach(), out={k: now[k].detach() for k in FIELDS}, grad={k: start[k].grad for k in FIELDS})
    with torch.no_grad():
        if kind == "step":
            new, co = ex.step(f, case)
            return dict(new, dt=co["dt"], alpha_si=co["alpha_si"])
        co = ex.coeffs(f)
        v = torch.stack([f["vr"], f["vt"], f["vp"]])
        b = ex.force(v, f["br"], f["bt"], f["bp"], co["dt"])
        f["br"], f["bt"], f["bp"] = ex.induction(v, case["eta"], co["dt"], f["br"], f["bt"], f["bp"])
        return dict(f, b=b, **co, **ex.diagnostics(f))
