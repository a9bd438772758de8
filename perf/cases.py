"""The work that a user of the library has it do, as cases to be timed.

Every pass goes through the public entry points (paper_2002_04222_gb300):
  residual  one evaluation of R(u) = M^-1 L(u, t), the call behind every
            Jacobian-free product, Newton residual and explicit update;
  apply     one BRJ(7) preconditioner application, the call made once per
            GMRES iteration;
  build     a rebuild in place of the BRJ blocks at a new state, and the first
            application of them (a user rebuilds every few steps);
  step      one implicit time step from u^n with a frozen preconditioner.
The Jacobian-free product and GMRES run inside the steps: a finite difference
divides the residual's rounding by 1e-8, so on their own their outputs hold
seven digits only.

The flows are those of the repository's workloads: the isentropic vortex and
the Poiseuille channel on quadrilaterals, the shock / boundary-layer
interaction with shock capturing, the Taylor-Green box, boxes of unequal
element counts and spacings, and the curved O-grid around a cylinder.
"""
import functools
import math

import numpy as np
import torch

import paper_2002_04222_gb300 as dgl
import workloads as w

LAMBDA = 1.0 - math.sqrt(0.5)        # diagonal of the two-stage SDIRK tableau


def listed():
    return [
        # the smallest call: the 8x8 vortex, where launches and latency are all there is
        dict(name="residual_vortex8_P2", kind="residual", flow="vortex", nx=8, P=2),
        # a wall-bounded channel at high order: Dirichlet, isothermal walls, forcing
        dict(name="residual_channel16x8_P5", kind="residual", flow="channel", nx=16, ny=8, P=5),
        # supersonic flow with shock capturing, adiabatic wall and far field
        dict(name="residual_swbli119x39_P3", kind="residual", flow="swbli", nx=119, ny=39, P=3),
        # an odd, stretched box with Sutherland's law and the HLLC flux
        dict(name="residual_box13x11x7_P2", kind="residual", flow="box", nx=13, ny=11, nz=7, P=2,
             riemann=1, mu_law=1),
        # the benchmark mesh, and the larger one at the next order
        dict(name="residual_tgv16_P3", kind="residual", flow="tgv", nx=16, P=3),
        dict(name="residual_tgv24_P4", kind="residual", flow="tgv", nx=24, P=4),
        # curved quadratic elements around a cylinder
        dict(name="residual_cylinder_P3", kind="residual", flow="cylinder", nx=24, ny=48, nz=6, P=3),
        # the preconditioner of the benchmark step (FP32 blocks, one kernel per sweep, graphs)
        dict(name="apply_tgv16_P3_fp32", kind="apply", flow="tgv", nx=16, P=3, precision="fp32"),
        # BF16 blocks on the curved mesh, as the cylinder run uses them
        dict(name="apply_cylinder_P3_bf16", kind="apply", flow="cylinder", nx=12, ny=24, nz=6, P=3,
             precision="bf16"),
        # rebuilding the blocks at a new state
        dict(name="build_tgv10_P3_fp32", kind="build", flow="tgv", nx=10, P=3, precision="fp32"),
        # whole steps: the small vortex with the defaults (FP64 blocks), the benchmark's step
        dict(name="step_vortex8_P2_fp64", kind="step", flow="vortex", nx=8, P=2, precision="fp64"),
        dict(name="step_tgv16_P3_fp32", kind="step", flow="tgv", nx=16, P=3, precision="fp32"),
    ]


def _log(rng, a, b):
    return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))


def draw(rng):
    kind = rng.choice(["residual", "residual", "residual", "residual", "apply", "build", "step"])
    if kind == "residual":
        flow = rng.choice(["vortex", "channel", "swbli", "box", "tgv", "cylinder"])
        if flow == "vortex":
            return dict(kind=kind, flow=flow, nx=_log(rng, 5, 96), P=rng.randint(1, 6),
                        riemann=rng.choice([0, 0, 1, 2, 3, 4]), mu_law=rng.choice([0, 1]))
        if flow == "channel":
            return dict(kind=kind, flow=flow, nx=_log(rng, 8, 96), ny=2 * _log(rng, 3, 24),
                        P=rng.randint(1, 6))
        if flow == "swbli":
            return dict(kind=kind, flow=flow, nx=_log(rng, 30, 160), ny=_log(rng, 11, 60),
                        P=rng.randint(2, 4), av=rng.choice([1, 1, 2]))
        if flow == "box":
            return dict(kind=kind, flow=flow, nx=_log(rng, 3, 22), ny=_log(rng, 3, 22),
                        nz=_log(rng, 2, 22), P=rng.randint(1, 4), riemann=rng.choice([0, 0, 1]),
                        mu_law=rng.choice([0, 1]))
        if flow == "tgv":
            return dict(kind=kind, flow=flow, nx=_log(rng, 4, 22), P=rng.randint(1, 4))
        return dict(kind=kind, flow=flow, nx=_log(rng, 6, 28), ny=_log(rng, 12, 48),
                    nz=rng.randint(2, 7), P=rng.randint(1, 3))
    if kind == "apply":
        flow = rng.choice(["tgv", "box", "vortex", "cylinder"])
        if flow == "vortex":
            return dict(kind=kind, flow=flow, nx=_log(rng, 6, 64), P=rng.randint(2, 5),
                        precision=rng.choice(["fp64", "fp32", "bf16"]))
        if flow == "cylinder":
            return dict(kind=kind, flow=flow, nx=_log(rng, 5, 12), ny=_log(rng, 12, 24),
                        nz=rng.randint(2, 6), P=rng.randint(2, 3),
                        precision=rng.choice(["fp32", "bf16"]))
        return dict(kind=kind, flow=flow, nx=_log(rng, 3, 14), ny=_log(rng, 3, 14),
                    nz=_log(rng, 3, 14), P=rng.randint(2, 3),
                    precision=rng.choice(["fp32", "fp32", "bf16", "fp64"]))
    if kind == "build":
        if rng.random() < 0.5:
            return dict(kind=kind, flow="vortex", nx=_log(rng, 6, 40), P=rng.randint(2, 4),
                        precision=rng.choice(["fp64", "fp32"]))
        return dict(kind=kind, flow="box", nx=_log(rng, 3, 10), ny=_log(rng, 3, 10),
                    nz=_log(rng, 3, 10), P=rng.randint(2, 3), precision=rng.choice(["fp32", "bf16"]))
    if rng.random() < 0.5:
        return dict(kind=kind, flow="vortex", nx=_log(rng, 5, 32), P=rng.randint(2, 4),
                    precision=rng.choice(["fp64", "fp32"]))
    return dict(kind=kind, flow="tgv", nx=_log(rng, 4, 14), P=rng.randint(2, 3),
                precision=rng.choice(["fp32", "fp32", "bf16"]))


# ------------------------------------------------------------------ inputs
@functools.lru_cache(maxsize=16)
def _flow(flow, nx, ny, nz, P, riemann, mu_law, av):
    """The workload (mesh, orders, physics); meshes are a user's own files."""
    if flow == "vortex":
        c = w.vortex_case(n=nx, P=P)
    elif flow == "channel":
        c = w.poiseuille_case(P, nx=nx, ny=ny, ratio=1.1 if ny <= 16 else 1.04)
    elif flow == "swbli":
        c = w.swbli_case(nx=nx, ny=ny, P=P, av=av or 1)
    elif flow == "box":
        c = w.small_tgv_case((nx, ny, nz), P=P, stretch=True)
    elif flow == "tgv":
        c = w.small_tgv_case((nx, ny or nx, nz or nx), P=P)
    else:
        c = w.cylinder_case(nx, ny, nz, P=P, wall_layer=0.1)
    if riemann:
        c.phys.riemann = riemann
    if mu_law:
        c.phys.mu_law = mu_law
    return c


def _workload(case):
    return _flow(case["flow"], case["nx"], case.get("ny", 0), case.get("nz", 0), case["P"],
                 case.get("riemann", 0), case.get("mu_law", 0), case.get("av", 0))


def _noise(shape, seed, device):
    g = torch.Generator(device=device).manual_seed(int(seed))
    return torch.randn(shape, dtype=torch.float64, device=device, generator=g)


def _perturbed(u, seed, amp):
    """The projected field plus seeded noise on every coefficient, amp x the
    RMS of density and energy and 5 amp x that of the momentum, every component
    alike: the jumps between elements, and the cross flow, of a flow under way."""
    rms = u.square().mean(dim=(0, 2), keepdim=True).sqrt()
    rms[:, 1:-1] = 5.0 * rms[:, 1:-1].square().mean().sqrt()
    return u + amp * rms * _noise(u.shape, seed, u.device)


def _dt(case, c):
    """The workloads' own rules: the Taylor-Green step at 10x the explicit one,
    0.01 for the small vortex (scaled with its element), the first radial
    cell's convective step for the cylinder."""
    if case["flow"] in ("tgv", "box"):
        return w.tgv_dt(max(case["nx"], case.get("ny", 0), case.get("nz", 0)), case["P"], c.phys.Ma)
    if case["flow"] == "vortex":
        return 0.01 * 8.0 / case["nx"]
    r = np.sqrt((c.mesh.nodes[..., :2] ** 2).sum(-1))
    return 1.7 * float((r.max(1) - r.min(1)).min()) / case["P"]


def _opts(case):
    """The options that the benchmark sets; FP64 blocks are the library's defaults."""
    if case["precision"] == "fp64":
        return dict(precision="fp64")
    return dict(precision=case["precision"], graphs=True, fused=True)


def prepare(case, seed):
    c = _workload(case)
    m = dgl.Mesh.from_case(c)
    dgl.apply_tuning(m)
    s = {"kind": case["kind"], "mesh": m, "opts": None}
    u0 = m.project(0.0)
    if case["kind"] == "residual":
        s["u"] = _perturbed(u0, seed, 1e-2)
        s["out"] = m.empty()
        return s
    dt = _dt(case, c)
    # (a step starts from the end of the one before: small jumps)
    s["u"] = _perturbed(u0, seed, 2e-4 if case["kind"] == "step" else 1e-3)
    s["out"] = m.empty()
    s["opts"] = _opts(case)
    s["dt"] = dt
    s["pc"] = dgl.Precond(m).build(s["u"], 0.0, LAMBDA * dt, **s["opts"])
    if case["kind"] == "step":
        s["opts"] = dict(precision=case["precision"], graphs=case["precision"] != "fp64",
                         fused=case["precision"] != "fp64")
    else:
        s["q"] = _noise(u0.shape, seed + 1_000_003, u0.device)
    if case["kind"] == "build":
        s["u"] = _perturbed(u0, seed + 2_000_003, 1e-3)     # the state of the rebuild
    return s


def run(s):
    m = s["mesh"]
    if s["kind"] == "residual":
        return m.residual(s["u"], 0.0, out=s["out"])
    if s["kind"] == "apply":
        return s["pc"].apply(s["q"], out=s["out"])
    if s["kind"] == "build":
        s["pc"].build(s["u"], 0.0, LAMBDA * s["dt"], **s["opts"])
        return s["pc"].apply(s["q"], out=s["out"])
    s["out"].copy_(s["u"])
    m.sdirk_step(s["out"], 0.0, s["dt"], precond=s["pc"], restart=30, **s["opts"])
    return s["out"]


# ------------------------------------------------------------------ work
def _residual_flops(d, P, Q, E, F):
    """Sum-factorised operation count (a multiply-add as 2) of one residual."""
    n, nv = P + 1, d + 2
    fwd = sum(n ** (d - k) * Q ** (k + 1) for k in range(d))          # modes to points
    line = Q ** (d + 1)                                             # one direction, all points
    per = 2 * nv * (2 * fwd + 2 * d * line + 2 * 2 * d * (1 + d) * line // Q)
    return E * (per + (190 if d == 3 else 110) * Q ** d) + F * Q ** (d - 1) * (420 if d == 3 else 260)


def work(case):
    c = _workload(case)
    d, P, Q, E, F = c.mesh.dim, c.P, c.Q, c.mesh.n_elem, c.mesh.n_faces
    nb = (d + 2) * (P + 1) ** d
    vec = 8.0 * E * nb
    geom = 8.0 * c.mesh.nodes.size
    res = _residual_flops(d, P, Q, E, F)
    if case["kind"] == "residual":
        return {"bytes": 2 * vec + geom, "flops": res}
    size = {"fp64": 8, "fp32": 4, "bf16": 2}[case["precision"]]
    blocks = float(E) * nb * nb * size
    jac = float(E) * 2 * d * Q ** (d - 1) * (d + 2) ** 2 * (8 if size == 8 else 4)
    sweeps = 7 * 2.0 * E * nb * nb
    if case["kind"] == "apply":
        return {"bytes": blocks + jac + 2 * vec, "flops": sweeps}
    if case["kind"] == "build":
        return {"bytes": blocks + jac + 3 * vec, "flops": 2.0 * E * nb ** 3 + sweeps + res}
    # a step of two stages needs at least one Newton iteration with one product
    # and one preconditioner application in each, and three residuals
    return {"bytes": blocks + jac + 2 * vec, "flops": 8 * res + 4 * sweeps}


# ------------------------------------------------------------------ 64-bit values
def exact(case, seed):
    """The residual and the BRJ application in plain torch, 64 bits, dense
    per-element operators.  A step has no such value: Newton and GMRES stop at
    their tolerances, and what they stop at is the step's result."""
    if case["kind"] == "step":
        return None
    c = _workload(case)
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    m = dgl.Mesh.from_case(c)
    u0 = m.project(0.0)
    m.close()
    ref = _Plain(c, dev)
    if case["kind"] == "residual":
        return ref.residual(_perturbed(u0, seed, 1e-2))
    amp_seed = seed + 2_000_003 if case["kind"] == "build" else seed
    u = _perturbed(u0, amp_seed, 1e-3)
    q = _noise(u0.shape, seed + 1_000_003, u0.device)
    return ref.brj(u, q, LAMBDA * _dt(case, c))


def _prim(U, ph):
    d = U.shape[-1] - 2
    v = U[..., 1:1 + d] / U[..., :1]
    p = (ph.gamma - 1) * (U[..., -1] - 0.5 * (U[..., 1:1 + d] * v).sum(-1))
    return U[..., 0], v, p


def _cons(rho, v, p, ph):
    return torch.cat([rho[..., None], rho[..., None] * v,
                      (p / (ph.gamma - 1) + 0.5 * rho * (v * v).sum(-1))[..., None]], -1)


def _euler(U, ph):
    """Advection flux [..., i, v]."""
    d = U.shape[-1] - 2
    _, v, p = _prim(U, ph)
    F = v[..., :, None] * U[..., None, :]
    F = F + p[..., None, None] * torch.eye(d, d + 2, dtype=U.dtype, device=U.device).roll(1, -1)
    return F + torch.cat([torch.zeros_like(F[..., :-1]), (p[..., None] * v)[..., None]], -1)


def _mu(U, ph):
    rho, _, p = _prim(U, ph)
    if ph.mu_law == 0:
        return torch.full_like(p, 1.0 / ph.Re)
    T, s = ph.gamma * ph.Ma ** 2 * p / rho, 110.0 / ph.T_inf_K
    return T ** 1.5 * (1 + s) / (T + s) / ph.Re


def _viscous(U, dU, ph, mu):
    """Diffusion flux [..., i, v] for the gradient dU[..., j, v]."""
    d = U.shape[-1] - 2
    rho, v, _ = _prim(U, ph)
    dr = dU[..., 0]
    dv = (dU[..., 1:1 + d] - v[..., None, :] * dr[..., None]) / rho[..., None, None]   # [j, k]
    de = (dU[..., -1] - (U[..., -1] / rho)[..., None] * dr) / rho[..., None]
    dT = ph.gamma * ph.Ma ** 2 * (ph.gamma - 1) * (de - (dv * v[..., None, :]).sum(-1))
    div = dv.diagonal(dim1=-2, dim2=-1).sum(-1)
    eye = torch.eye(d, dtype=U.dtype, device=U.device)
    tau = mu[..., None, None] * (dv + dv.transpose(-1, -2) - 2.0 / 3.0 * div[..., None, None] * eye)
    en = (tau * v[..., None, :]).sum(-1) + (mu / (ph.Ma ** 2 * ph.Pr * (ph.gamma - 1)))[..., None] * dT
    return torch.cat([torch.zeros_like(dr)[..., None], tau, en[..., None]], -1)


def _av(U, fac, ph):
    """mu_av = f_e rho (c + |u|)."""
    rho, v, p = _prim(U, ph)
    return fac * rho * ((ph.gamma * p / rho).sqrt() + v.norm(dim=-1))


def _ducros(U, dU):
    d = U.shape[-1] - 2
    v = U[..., 1:1 + d] / U[..., :1]
    dv = (dU[..., 1:1 + d] - v[..., None, :] * dU[..., :1]) / U[..., :1, None]
    div2 = dv.diagonal(dim1=-2, dim2=-1).sum(-1) ** 2
    a = dv - dv.transpose(-1, -2)
    return div2 / (div2 + 0.5 * (a * a).sum((-1, -2)) + 1e-6)


def _riemann(UL, UR, n, ph):
    g = ph.gamma
    rL, vL, pL = _prim(UL, ph)
    rR, vR, pR = _prim(UR, ph)
    unL, unR = (vL * n).sum(-1), (vR * n).sum(-1)
    FL = (_euler(UL, ph) * n[..., None]).sum(-2)
    FR = (_euler(UR, ph) * n[..., None]).sum(-2)
    cL, cR = (g * pL / rL).sqrt(), (g * pR / rR).sqrt()
    if ph.riemann == w.RIEMANN_LF:
        lam = torch.maximum(unL.abs() + cL, unR.abs() + cR)
        return 0.5 * (FL + FR) - 0.5 * lam[..., None] * (UR - UL)
    if ph.riemann == w.RIEMANN_AUSM:
        ML, MR = unL / cL, unR / cR
        Mp = torch.where(ML.abs() <= 1, 0.25 * (ML + 1) ** 2, 0.5 * (ML + ML.abs()))
        Mm = torch.where(MR.abs() <= 1, -0.25 * (MR - 1) ** 2, 0.5 * (MR - MR.abs()))
        Pp = torch.where(ML.abs() <= 1, 0.25 * (ML + 1) ** 2 * (2 - ML), 0.5 * (1 + ML.sign()))
        Pm = torch.where(MR.abs() <= 1, 0.25 * (MR - 1) ** 2 * (2 + MR), 0.5 * (1 - MR.sign()))
        m = (Mp + Mm)[..., None]
        pp = torch.zeros_like(UL)
        pp[..., 1:-1] = (Pp * pL + Pm * pR)[..., None] * n
        hL, hR = UL.clone(), UR.clone()
        hL[..., -1] += pL
        hR[..., -1] += pR
        hL, hR = cL[..., None] * hL, cR[..., None] * hR
        return 0.5 * m * (hL + hR) - 0.5 * m.abs() * (hR - hL) + pp
    sL, sR = rL.sqrt(), rR.sqrt()
    HL, HR = (UL[..., -1] + pL) / rL, (UR[..., -1] + pR) / rR
    ut = (sL[..., None] * vL + sR[..., None] * vR) / (sL + sR)[..., None]
    Ht = (sL * HL + sR * HR) / (sL + sR)
    q2 = (ut * ut).sum(-1)
    c2 = (g - 1) * (Ht - 0.5 * q2)
    c, un = c2.sqrt(), (ut * n).sum(-1)
    if ph.riemann == w.RIEMANN_ROE:
        rt, dp, du = sL * sR, pR - pL, vR - vL
        dun = (du * n).sum(-1)
        w1 = (un - c).abs() * (dp - rt * c * dun) / (2 * c2)
        w5 = (un + c).abs() * (dp + rt * c * dun) / (2 * c2)
        w2, ws = un.abs() * (rR - rL - dp / c2), un.abs() * rt
        mom = (w1 + w5 + w2)[..., None] * ut + ((w5 - w1) * c)[..., None] * n + \
            ws[..., None] * (du - dun[..., None] * n)
        en = (w1 + w5) * Ht + (w5 - w1) * un * c + 0.5 * w2 * q2 + ws * ((ut * du).sum(-1) - un * dun)
        return 0.5 * (FL + FR) - 0.5 * torch.cat([(w1 + w2 + w5)[..., None], mom, en[..., None]], -1)
    SL, SR = torch.minimum(unL - cL, un - c), torch.maximum(unR + cR, un + c)
    if ph.riemann == w.RIEMANN_HLL:
        Fm = (SR[..., None] * FL - SL[..., None] * FR + (SL * SR)[..., None] * (UR - UL)) / (SR - SL)[..., None]
        return torch.where((SL >= 0)[..., None], FL, torch.where((SR <= 0)[..., None], FR, Fm))
    Ss = (pR - pL + rL * unL * (SL - unL) - rR * unR * (SR - unR)) / (rL * (SL - unL) - rR * (SR - unR))

    def star(U, r, v, p, u, S, F):
        f = r * (S - u) / (S - Ss)
        m = f[..., None] * (v + (Ss - u)[..., None] * n)
        e = f * (U[..., -1] / r + (Ss - u) * (Ss + p / (r * (S - u))))
        return F + S[..., None] * (torch.cat([f[..., None], m, e[..., None]], -1) - U)

    a, b = star(UL, rL, vL, pL, unL, SL, FL), star(UR, rR, vR, pR, unR, SR, FR)
    return torch.where((SL >= 0)[..., None], FL, torch.where((Ss >= 0)[..., None], a,
                       torch.where((SR > 0)[..., None], b, FR)))


def _field(ph, x):
    """The analytic states that the boundaries of these flows take, at t = 0."""
    d, g, Ma = x.shape[-1], ph.gamma, ph.Ma
    rho = torch.ones_like(x[..., 0])
    v, T = torch.zeros_like(x), torch.ones_like(rho)
    if ph.fid == w.FIELD_POISEUILLE:
        theta, L, dp = ph.fpar
        y = x[..., 1]
        v[..., 0] = -0.5 * dp * ph.Re * (y * (L - y) + theta * y * y * (L - y) ** 2)
        T = 1.0 + g * Ma ** 2 * dp * x[..., 0]
    elif ph.fid == w.FIELD_SHOCK:
        b, xs, width, layer = math.radians(ph.fpar[0]), ph.fpar[1], ph.fpar[2], ph.fpar[3]
        sb, cb = math.sin(b), math.cos(b)
        mn2 = (Ma * sb) ** 2
        r2 = (g + 1) * mn2 / ((g - 1) * mn2 + 2)
        p2 = 1 + 2 * g / (g + 1) * (mn2 - 1)
        post = 0.5 * (1 + torch.tanh((x[..., 1] * cb - (xs - x[..., 0]) * sb) / width))
        rho = 1 + post * (r2 - 1)
        v[..., 0] = 1 + post * (sb * sb / r2 + cb * cb - 1)
        v[..., 1] = post * (sb / r2 * cb - cb * sb)
        v = v * (1 - torch.exp(-x[..., 1] / layer))[..., None]
        T = (1 + post * (p2 - 1)) / rho
    else:                                  # the cylinder's stream, at rest on its wall
        v[..., 0] = 1 - torch.exp(-(x[..., :2].norm(dim=-1) - ph.fpar[0]).clamp(min=0) / ph.fpar[1])
    return _cons(rho, v, rho * T / (g * Ma ** 2), ph)


def _boundary(ph, kind, x, UL, n):
    """(exterior state of the Riemann flux, state of the viscous flux)."""
    g = ph.gamma
    rho, v, p = _prim(UL, ph)
    if kind == w.BC_ADIA_WALL:
        return (_cons(rho, v - 2 * (v * n).sum(-1, keepdim=True) * n, p, ph),
                _cons(rho, torch.zeros_like(v), p, ph))
    if kind == w.BC_ISO_WALL:
        Tw = 1.0 + g * ph.Ma ** 2 * ph.fpar[2] * x[..., 0]
        B = _cons(rho, torch.zeros_like(v), rho * Tw / (g * ph.Ma ** 2), ph)
        return B, B
    B = _field(ph, x)
    if kind == w.BC_FARFIELD:
        ri, vi, pi = _prim(B, ph)
        c, ci = (g * p / rho).sqrt(), (g * pi / ri).sqrt()
        un, ui = (v * n).sum(-1), (vi * n).sum(-1)
        Rp, Rm = un + 2 * c / (g - 1), ui - 2 * ci / (g - 1)
        ub, cb = 0.5 * (Rp + Rm), 0.25 * (g - 1) * (Rp - Rm)
        out = ub > 0
        s = torch.where(out, p / rho ** g, pi / ri ** g)
        vu = torch.where(out[..., None], v, vi)
        vt = vu - (vu * n).sum(-1, keepdim=True) * n
        rb = (cb * cb / (g * s)) ** (1 / (g - 1))
        A = _cons(rb, vt + ub[..., None] * n, rb * cb * cb / g, ph)
        B = torch.where((un >= c)[..., None], UL, torch.where((un <= -c)[..., None], B, A))
    return B, B


def _basis(P, x):
    """Modified basis and its derivative at x: two numpy arrays [len(x)][P+1]."""
    from numpy.polynomial import polynomial as pl
    polys = [np.array([0.5, -0.5])]
    jac = [np.array([1.0]), np.array([0.0, 2.0])]                # P_k^(1,1)
    for k in range(1, P):
        a1, a3, a4 = 2 * (k + 1) * (k + 3) * (2 * k + 2), (2 * k + 2) * (2 * k + 3) * (2 * k + 4), \
            2 * (k + 1) ** 2 * (2 * k + 4)
        jac.append(pl.polysub(a3 * np.concatenate([[0.0], jac[k]]), a4 * jac[k - 1]) / a1)
    polys += [pl.polymul([0.25, 0.0, -0.25], jac[k]) for k in range(P - 1)] + [np.array([0.5, 0.5])]
    return (np.stack([pl.polyval(x, p) for p in polys], 1),
            np.stack([pl.polyval(x, pl.polyder(p)) for p in polys], 1))


def _tensor(tabs):
    """Tensor product of 1-D tables [np][nm], first direction fastest."""
    out = np.ones((1, 1))
    for t in tabs:
        out = np.kron(t, out)
    return out


class _Plain:
    """Dense per-element operators of one workload in 64 bits."""

    def __init__(self, c, dev):
        self.ph, mesh, P, Q = c.phys, c.mesh, c.P, c.Q
        self.P, self.d, self.dev = P, mesh.dim, dev
        d, g = self.d, mesh.geom_order
        xq, wq = np.polynomial.legendre.leggauss(Q)
        t = functools.partial(torch.as_tensor, dtype=torch.float64, device=dev)
        nodes = t(mesh.nodes)
        gx = np.linspace(-1, 1, g + 1)

        def tables(pts):
            """Basis B, dB[r] and mapped points, metrics at a tensor grid of points."""
            b = [_basis(P, p) for p in pts]
            V = np.linalg.inv(np.vander(gx, increasing=True))
            s = [(np.vander(p, g + 1, increasing=True) @ V,
                  np.stack([k * p ** max(k - 1, 0) for k in range(g + 1)], 1) @ V) for p in pts]
            B = t(_tensor([x[0] for x in b]))
            dB = t(np.stack([_tensor([x[r == k] for k, x in enumerate(b)]) for r in range(d)]))
            S = t(_tensor([x[0] for x in s]))
            dS = t(np.stack([_tensor([x[r == k] for k, x in enumerate(s)]) for r in range(d)]))
            X = torch.einsum("qa,eax->eqx", S, nodes)
            J = torch.einsum("rqa,eax->eqxr", dS, nodes)
            return B, dB, X, torch.linalg.inv(J), torch.linalg.det(J)

        self.B, self.dB, self.x, self.gi, det = tables([xq] * d)
        self.wref = t(_tensor([wq[:, None]] * d)[:, 0])
        self.wJ = self.wref * det
        vol = self.wJ.sum(1)
        self.h = vol ** (1.0 / d)
        self.M = torch.einsum("qm,eq,qn->emn", self.B, self.wJ, self.B)
        if self.ph.av:                      # projection onto degree <= P-1 of the sensor
            L = np.stack([np.polynomial.legendre.legval(xq, np.eye(P)[k]) for k in range(P)], 1)
            p1 = L @ np.linalg.solve(L.T @ (wq[:, None] * L), L.T * wq)
            self.Pi = t(_tensor([p1] * d))
        faces = torch.as_tensor(mesh.faces, device=dev).long()
        sides = [tables([np.array([2.0 * (lf % 2) - 1]) if r == lf // 2 else xq for r in range(d)])
                 for lf in range(2 * d)]
        wf = t(_tensor([wq[:, None]] * (d - 1))[:, 0])
        self.groups = []
        key = (faces[:, 1] * 64 + (faces[:, 3] + 1)) * 64 + faces[:, 5] + 1
        for k in key.unique().tolist():
            f = faces[key == k]
            lf, rf, bc = int(f[0, 1]), int(f[0, 3]), int(f[0, 5])
            e = f[:, 0]
            Bf, dBf, X, gi, dj = sides[lf]
            nrm = gi[e][:, :, lf // 2] * (2 * (lf % 2) - 1)
            mag = nrm.norm(dim=-1)
            G = dict(e=[e], B=[Bf], dB=[dBf], gi=[gi[e]], n=nrm / mag[..., None], x=X[e],
                     w=wf * dj[e].abs() * mag, bc=None)
            area = G["w"].sum(1)
            h = vol[e] / area
            if rf >= 0:
                r = f[:, 2]
                for name, v in zip(("e", "B", "dB", "gi"), (r, sides[rf][0], sides[rf][1], sides[rf][3][r])):
                    G[name].append(v)
                h = torch.minimum(h, vol[r] / area)
            else:
                G["bc"] = self.ph.bc[bc]
            G["beta"] = (P + 1) ** 2 / h
            self.groups.append(G)

    def _grad(self, u, dB, gi):
        return torch.einsum("eqrj,reqv->eqjv", gi, torch.einsum("rqm,evm->reqv", dB, u))

    def _factor(self, u):
        ph = self.ph
        rho = torch.einsum("qm,em->eq", self.B, u[:, 0])
        dr = rho - rho @ self.Pi.T
        s = torch.log10((dr * dr) @ self.wref / ((rho * rho) @ self.wref))
        s0, k = -4 * math.log10(self.P), ph.av_kappa
        ramp = 0.5 * (1 + torch.sin(0.5 * math.pi * (s - s0).clamp(-k, k) / k))
        S = torch.where(s < s0 - k, torch.zeros_like(s), torch.where(s > s0 + k, torch.ones_like(s), ramp))
        return ph.av_mu0 * S * self.h / self.P

    def _volume(self, U, dU, mua):
        H = _euler(U, self.ph)
        return H - _viscous(U, dU, self.ph, _mu(U, self.ph) + mua) if self.ph.viscous else H

    def _traces(self, G, u):
        q = [torch.einsum("pm,evm->epv", B, u[e]) for e, B in zip(G["e"], G["B"])]
        dq = [self._grad(u[e], dB, gi) for e, dB, gi in zip(G["e"], G["dB"], G["gi"])]
        return q, sum(dq) / len(dq)

    def _face_mu(self, G, q, dqa, fac):
        if fac is None:
            return 0.0
        a = sum(_av(x, fac[e][:, None], self.ph) for x, e in zip(q, G["e"])) / len(q)
        return a * _ducros(sum(q) / len(q), dqa) if self.ph.av == 2 else a

    def _flux(self, G, q, dqa, mua):
        """H^n and the symmetric flux S[i] at the face points."""
        ph, n = self.ph, G["n"]
        if G["bc"] is None:
            ext, Qa, jump = q[1], 0.5 * (q[0] + q[1]), q[0] - q[1]
        else:
            ext, Qa = _boundary(ph, G["bc"], G["x"], q[0], n)
            jump = q[0] - Qa
        H = _riemann(q[0], ext, n, ph)
        if not ph.viscous:
            return H, None
        mu = _mu(Qa, ph) + mua
        S = _viscous(Qa, n[..., :, None] * jump[..., None, :], ph, mu)
        Gn = (n[..., None] * (_viscous(Qa, dqa, ph, mu) - G["beta"][:, None, None, None] * S)).sum(-2)
        if G["bc"] == w.BC_ADIA_WALL:
            keep = torch.ones(S.shape[-1], dtype=S.dtype, device=S.device)
            keep[-1] = 0
            Gn, S = Gn * keep, S * keep
        return H - Gn, S

    def residual(self, u):
        ph = self.ph
        fac = self._factor(u) if ph.av else None
        L = torch.empty_like(u)
        step = max(1, 2_000_000 // self.B.shape[0])
        for a in range(0, u.shape[0], step):
            s = slice(a, a + step)
            U, dU = torch.einsum("qm,evm->eqv", self.B, u[s]), self._grad(u[s], self.dB, self.gi[s])
            mua = 0.0
            if fac is not None:
                mua = _av(U, fac[s][:, None], ph) * (_ducros(U, dU) if ph.av == 2 else 1.0)
            H = torch.einsum("eqrj,eqjv->eqrv", self.gi[s], self._volume(U, dU, mua)) * self.wJ[s][..., None, None]
            L[s] = torch.einsum("rqm,eqrv->evm", self.dB, H)
            if ph.forcing:
                theta, Ly, dp = ph.fpar
                y, mu = self.x[s][..., 1], 1.0 / ph.Re
                cc = Ly * Ly - 6 * y * Ly + 6 * y * y
                hh = y * (Ly - y) + theta * y * y * (Ly - y) ** 2
                f = torch.zeros_like(U)
                f[..., 1] = dp * theta * cc
                f[..., -1] = dp ** 2 / (2 * mu) * hh * (1 - theta * cc - ph.gamma / (ph.gamma - 1)) - \
                    dp ** 2 / (4 * mu) * (Ly - 2 * y) ** 2 * (2 * theta * y * (Ly - y) + 1) ** 2
                L[s] += torch.einsum("qm,eqv->evm", self.B, f * self.wJ[s][..., None])
        for G in self.groups:
            q, dqa = self._traces(G, u)
            H, S = self._flux(G, q, dqa, self._face_mu(G, q, dqa, fac))
            H, sgn = H * G["w"][..., None], -1.0
            for e, B, dB, gi in zip(G["e"], G["B"], G["dB"], G["gi"]):
                add = sgn * torch.einsum("pm,fpv->fvm", B, H)
                if S is not None:
                    add += ph.beta_s / len(G["e"]) * torch.einsum(
                        "rpm,fprj,fpjv->fvm", dB, gi, S * G["w"][..., None, None])
                L.index_add_(0, e, add)
                sgn = 1.0
        return torch.linalg.solve(self.M, L.transpose(1, 2)).transpose(1, 2).contiguous()

    def brj(self, u, q, dta, J=7):
        """q^J of the block relaxed Jacobi iteration, omega = 1."""
        ph, (E, nv, nm), d = self.ph, u.shape, self.d
        A = torch.empty((E, nv, nm, nv, nm), dtype=torch.float64, device=u.device)
        unit = torch.eye(nv, dtype=torch.float64, device=u.device)
        step = max(1, 60_000 // self.B.shape[0])
        for a in range(0, E, step):
            s = slice(a, a + step)
            U, dU = torch.einsum("qm,evm->eqv", self.B, u[s]), self._grad(u[s], self.dB, self.gi[s])
            DB = torch.einsum("eqrj,rqm->ejqm", self.gi[s], self.dB)
            for l in range(nv):
                dv = unit[l].expand_as(U)
                _, A0 = torch.func.jvp(lambda x: self._volume(x, dU, 0.0), (U,), (dv,))
                X = torch.einsum("eqjk,qn->eqjkn", A0, self.B)
                for i in range(d if ph.viscous else 0):
                    gu = torch.zeros_like(dU)
                    gu[..., i, l] = 1.0
                    X -= torch.einsum("eqjk,eqn->eqjkn", _viscous(U, gu, ph, _mu(U, ph)), DB[:, i])
                A[s, :, :, l] = torch.einsum("ejqm,eq,eqjkn->ekmn", DB, self.wJ[s], X)
        chi = 2.0 ** -26 * u.square().sum(dim=(0, 2)).sqrt()
        off = []
        for G in self.groups:
            tr, dqa = self._traces(G, u)
            H0, _ = self._flux(G, tr, dqa, 0.0)
            jac = []
            for side in range(len(tr)):
                cols = []
                for l in range(nv):
                    p = list(tr)
                    p[side] = tr[side] + chi[l] * unit[l]
                    cols.append((self._flux(G, p, dqa, 0.0)[0] - H0) / chi[l])
                jac.append(torch.stack(cols, -1) * G["w"][..., None, None])          # [f][p][k][l]
            for side, sgn in zip(range(len(tr)), (-1.0, 1.0)):
                B = G["B"][side]
                A.index_add_(0, G["e"][side], sgn * torch.einsum("pm,fpkl,pn->fkmln", B, jac[side], B))
                if len(tr) == 2:
                    off.append((G["e"][side], G["e"][1 - side], B, G["B"][1 - side], sgn * jac[1 - side]))
        Mi = torch.linalg.inv(self.M)
        for a in range(0, E, 256):
            A[a:a + 256] = -dta * torch.einsum("emn,eknlo->ekmlo", Mi[a:a + 256], A[a:a + 256])
        D = A.view(E, nv * nm, nv * nm)
        D.diagonal(dim1=1, dim2=2).add_(1.0)
        lu, piv = torch.linalg.lu_factor(D)
        x = torch.zeros_like(q)
        for _ in range(J):
            y = torch.zeros_like(q)
            for e, o, B, Bo, Jo in off:
                y.index_add_(0, e, torch.einsum("pm,fpkl,pn,fln->fkm", B, Jo, Bo, x[o]))
            y = q + dta * torch.einsum("emn,evn->evm", Mi, y)
            x = torch.linalg.lu_solve(lu, piv, y.reshape(E, -1, 1)).view_as(q)
        return x
