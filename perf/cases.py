"""Performance cases of the library: what a coronal-model user has it compute.

Each case is one call (or one forward + backward) through the public Python
entry points of ``paper_2209_04481_gb300`` on seeded synthetic shells:

* ``residual``       R = dU/dt of one shell;
* ``gradient``       the differentiable residual, forward and backward;
* ``pseudo_time``    explicit pseudo-time steps of the FP64 master state;
* ``ensemble``       the residuals of many shells of different sizes at once;
* ``newton_krylov``  one implicit pseudo-time step;
* ``adjoint``        the magnetogram sensitivity of an outer functional.

``exact`` evaluates the same operator in plain float64 torch operations.
"""
import math
import random

import numpy as np
import torch

import coronal_inputs as ci
import paper_2209_04481_gb300 as pg

DEV = "cuda"
F64 = torch.float64
VR_STAR = 1935.07 / ci.V_REF   # prescribed inner outflow of the time-marching boundary
ANGULAR = ((24, 48), (48, 96), (96, 192))   # angular grids of the ensemble workload


def listed():
    return [
        # the smallest shell in use (pseudo-time and implicit test shell): launch and latency bound
        dict(name="residual_fp32_32x16x32", kind="residual", n_r=32, n_theta=16, n_phi=32,
             precision="fp32", limiter="vanalbada", inner_bc="low_e", state="wind"),
        # an odd shell whose rows and columns do not fill the tiles, the sharper limiter
        dict(name="residual_fp32_95x45x88", kind="residual", n_r=95, n_theta=45, n_phi=88,
             precision="fp32", limiter="minmod", inner_bc="low_e_wp", state="perturbed"),
        # the benchmark shell in the production precision
        dict(name="residual_fp32_128x64x128", kind="residual", n_r=128, n_theta=64, n_phi=128,
             precision="fp32", limiter="vanalbada", inner_bc="low_e", state="wind"),
        # the benchmark shell in plain FP64, with the norms and the step bound
        dict(name="residual_fp64_128x64x128", kind="residual", n_r=128, n_theta=64, n_phi=128,
             precision="fp64", limiter="vanalbada", inner_bc="low_e", state="wind"),
        # gradients through the residual on the benchmark shell (fitting a state)
        dict(name="gradient_fp32_128x64x128", kind="gradient", n_r=128, n_theta=64, n_phi=128,
             precision="fp32", limiter="vanalbada", inner_bc="low_e", state="perturbed"),
        # state and magnetogram gradients in FP64 on the adjoint workload's shell
        dict(name="gradient_fp64_64x32x64", kind="gradient", n_r=64, n_theta=32, n_phi=64,
             precision="fp64", limiter="vanalbada", inner_bc="low_e", state="perturbed"),
        # time marching on the benchmark shell: FP32 flux, FP64 master state, the
        # small CFL of a start from fields that are not yet in balance
        dict(name="pseudo_time_fp32_128x64x128", kind="pseudo_time", n_r=128, n_theta=64, n_phi=128,
             precision="fp32", limiter="vanalbada", inner_bc="low_e_wp", state="wind", steps=2, cfl=0.1),
        # time marching on a small FP64 shell: many short steps
        dict(name="pseudo_time_fp64_32x16x32", kind="pseudo_time", n_r=32, n_theta=16, n_phi=32,
             precision="fp64", limiter="vanalbada", inner_bc="low_e_wp", state="wind", steps=10, cfl=0.4),
        # eight shells of the ensemble workload's sizes in one call
        dict(name="ensemble_fp32_8", kind="ensemble", members=8, shapes_seed=5,
             precision="fp32", limiter="vanalbada", inner_bc="low_e_wp", state="wind"),
        # one implicit step of the production steady solve (line preconditioner, GMRES(60))
        dict(name="newton_krylov_fp64_96x48x96", kind="newton_krylov", n_r=96, n_theta=48, n_phi=96,
             precision="fp64", limiter="minmod", inner_bc="low_e_wp", state="wind", cfl=16.0,
             krylov_dim=60, precond=1),
        # one implicit step of the small steady solve (default options)
        dict(name="newton_krylov_fp64_32x16x32", kind="newton_krylov", n_r=32, n_theta=16, n_phi=32,
             precision="fp64", limiter="vanalbada", inner_bc="low_e_wp", state="wind", cfl=16.0,
             krylov_dim=30, precond=0),
        # magnetogram sensitivity of the mean outer density: a few accelerated adjoint passes
        dict(name="adjoint_fp64_32x16x32", kind="adjoint", n_r=32, n_theta=16, n_phi=32,
             precision="fp64", limiter="vanalbada", inner_bc="low_e_wp", state="wind", passes=4,
             krylov_dim=60, precond=1),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["residual", "residual", "residual", "gradient", "gradient", "pseudo_time",
                       "ensemble", "newton_krylov"])
    limiter = rng.choice(["vanalbada", "vanalbada", "minmod"])
    bc = rng.choice(["low_e", "low_e_wp"])
    if kind == "ensemble":
        return dict(kind=kind, members=rng.randint(3, 8), shapes_seed=rng.randint(0, 10 ** 6),
                    precision=rng.choice(["fp32", "fp32", "fp64"]), limiter=limiter, inner_bc="low_e_wp",
                    state="wind")
    shape = dict(n_r=_log_int(rng, 16, 144), n_theta=_log_int(rng, 10, 72),
                 n_phi=8 * _log_int(rng, 2, 18))
    state = rng.choice(["wind", "perturbed"])
    if kind == "residual":
        return dict(kind=kind, precision=rng.choice(["fp32", "fp32", "fp64"]), limiter=limiter,
                    inner_bc=bc, state=state, **shape)
    if kind == "gradient":
        # a perturbed state: the unperturbed wind sits on kinks of the flux
        return dict(kind=kind, precision=rng.choice(["fp32", "fp64"]), limiter="vanalbada",
                    inner_bc=bc, state="perturbed", **shape)
    if kind == "pseudo_time":
        precision = rng.choice(["fp32", "fp64"])
        steps, cfl = (rng.randint(1, 2), 0.1) if precision == "fp32" else (rng.randint(1, 12), 0.4)
        return dict(kind=kind, precision=precision, limiter=limiter, inner_bc="low_e_wp", state="wind",
                    steps=steps, cfl=cfl, **shape)
    return dict(kind=kind, n_r=_log_int(rng, 16, 64), n_theta=_log_int(rng, 10, 32),
                n_phi=8 * _log_int(rng, 2, 8), precision="fp64", limiter="vanalbada", inner_bc="low_e_wp",
                state="wind", cfl=rng.choice([2.0, 4.0, 8.0, 16.0]), krylov_dim=30,
                precond=rng.choice([0, 1]))


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _t(x):
    return torch.as_tensor(np.ascontiguousarray(x), dtype=F64, device=DEV)


def _shapes(case):
    if case["kind"] != "ensemble":
        return [(case["n_r"], case["n_theta"], case["n_phi"])]
    rng = random.Random(case["shapes_seed"])
    return [(rng.randint(48, 128),) + ANGULAR[m % 3] for m in range(case["members"])]


def _state(shape, kind, seed):
    """Parker wind with the aligned dipole, conservative (9, n_r, n_theta, n_phi).

    "wind": the primitives modulated by 2 % by a few smooth seeded modes, as a
    state on its way to steady; "perturbed": every primitive by 1 % seeded
    noise per cell."""
    gen = torch.Generator(device=DEV).manual_seed(seed)
    rc, tc, pc = (_t(x) for x in ci.cell_centres(*shape))
    R, T, P = rc[:, None, None], tc[None, :, None], pc[None, None, :]
    cs2 = ci.parker_sound_speed2()
    mach = _t(ci.parker_mach(rc.cpu().numpy()))[:, None, None]
    m_in = float(ci.parker_mach(np.array([ci.R_IN]))[0])
    one = torch.ones(shape, dtype=F64, device=DEV)
    v = mach * math.sqrt(cs2) * one
    rho = (m_in / mach) / R ** 2 * one
    st, ct, sp, cp = torch.sin(T), torch.cos(T), torch.sin(P), torch.cos(P)
    br, bt = ct / R ** 3, 0.5 * st / R ** 3
    W = torch.stack([rho, v * st * cp, v * st * sp, v * ct, (br * st + bt * ct) * cp * one,
                     (br * st + bt * ct) * sp * one, (br * ct - bt * st) * one, rho * cs2,
                     torch.zeros_like(rho)])
    bmag = torch.sqrt(W[4] ** 2 + W[5] ** 2 + W[6] ** 2)
    if kind == "perturbed":
        xi = torch.randn(W.shape, dtype=F64, device=DEV, generator=gen)
        W[:8] *= 1.0 + 0.01 * xi[:8]
        W[8] = 0.01 * xi[8] * bmag
    else:
        c = torch.randn((9, 3), dtype=F64, device=DEV, generator=gen)
        x, y, z = st * cp, st * sp, ct
        lr = torch.sin(1.5 * torch.log(R) + 0.5)
        for q in range(9):
            mode = (c[q, 0] * x * lr + c[q, 1] * y * z + c[q, 2] * z * lr) * one
            if q < 8:
                W[q] *= 1.0 + 0.02 * torch.tanh(mode)
            else:
                W[8] = 0.002 * mode * bmag
    rho, vx, vy, vz, bx, by, bz, p, psi = W
    E = p / (ci.GAMMA - 1.0) + 0.5 * rho * (vx * vx + vy * vy + vz * vz) + 0.5 * (bx * bx + by * by + bz * bz)
    return torch.stack([rho, rho * vx, rho * vy, rho * vz, bx, by, bz, E, psi])


def _magnetogram(shape, seed, amplitude):
    """cos(theta) + amplitude x the seeded multipoles (max |B_r| = 5 at amplitude 1)."""
    _, tc, pc = ci.cell_centres(2, shape[1], shape[2])
    dip = np.broadcast_to(np.cos(tc)[:, None], shape[1:])
    full = ci.magnetogram(shape[1], shape[2], lmax=min(15, shape[1] // 2), seed=seed)
    return _t(dip + amplitude * (full - dip))


def _inputs(case, seed):
    """[(shape, U in the grid's type (FP64 master state for time marching), B_r)] per shell."""
    implicit = case["kind"] in ("newton_krylov", "adjoint")
    master = implicit or case["kind"] == "pseudo_time"
    # strong fields where the state is only evaluated; where it is advanced, a
    # magnetogram near the state's own dipole
    amp = 0.05 if master else 1.0
    out = []
    for m, shape in enumerate(_shapes(case)):
        U = _state(shape, case["state"], seed + 1000 * m)
        if case["precision"] == "fp32" and not master:
            U = U.float()
        out.append((shape, U, _magnetogram(shape, seed + 1000 * m, amp)))
    return out


def prepare(case, seed):
    s = dict(case=case)
    grids, Us = [], []
    data = _inputs(case, seed)
    for shape, U, Br in data:
        g = pg.Grid(*shape, precision=case["precision"], limiter=case["limiter"], inner_bc=case["inner_bc"],
                    vr_star=VR_STAR, p_b=ci.parker_sound_speed2())
        g.set_inner_boundary(Br)
        grids.append(g)
        Us.append(U)
    s.update(grid=grids[0], U=Us[0], Br=data[0][2])
    if case["kind"] == "ensemble":
        s.update(grids=grids, Us=Us, Rs=[torch.empty_like(U) for U in Us], ens=pg.Ensemble(grids))
    elif case["kind"] == "residual":
        s.update(R=torch.empty_like(Us[0]))
        if case["precision"] == "fp64":
            s.update(norms=torch.empty(9, dtype=F64, device=DEV), dtmin=torch.empty(1, dtype=F64, device=DEV))
    elif case["kind"] == "gradient":
        gen = torch.Generator(device=DEV).manual_seed(seed + 4)
        s.update(Rbar=torch.randn(Us[0].shape, dtype=F64, device=DEV, generator=gen).to(Us[0].dtype))
        s["U"].requires_grad_(True)
        s["Br"].requires_grad_(case["precision"] == "fp64")
    else:
        s.update(U0=Us[0].clone())
        if case["kind"] == "adjoint":
            gbar = torch.zeros_like(Us[0])
            gbar[0, -1] = 1.0 / (case["n_theta"] * case["n_phi"])   # mean outer-layer density
            s.update(gbar=gbar, lam=torch.empty_like(gbar))
    torch.cuda.synchronize()
    return s


def run(s):
    case, g = s["case"], s["grid"]
    kind = case["kind"]
    if kind == "residual":
        R = g.residual(s["U"], s["R"], s.get("norms"), s.get("dtmin"))
        return dict(R=R, norms=s["norms"], dtmin=s["dtmin"]) if "norms" in s else dict(R=R)
    if kind == "gradient":
        R = pg.residual(s["U"], s["Br"], g)
        if s["Br"].requires_grad:
            Ubar, Brbar = torch.autograd.grad(R, (s["U"], s["Br"]), s["Rbar"])
            return dict(R=R, Ubar=Ubar, Brbar=Brbar)
        return dict(R=R, Ubar=torch.autograd.grad(R, s["U"], s["Rbar"])[0])
    if kind == "ensemble":
        return dict(R=s["ens"].residual(s["Us"], s["Rs"]))
    if kind == "adjoint":
        sens, lam, _ = g.adjoint_solve(s["U"], s["gbar"], s["lam"], krylov_dim=case["krylov_dim"],
                                       precond=case["precond"], lin_rtol=1e-8, adjoint_cfl=1000.0,
                                       adjoint_outer=case["passes"])
        return dict(sens=sens, lam=lam)
    # time marching starts each pass from the same state
    s["U"].copy_(s["U0"])
    if kind == "pseudo_time":
        g.pseudo_time_step(s["U"], case["steps"], case["cfl"])
        return dict(U=s["U"])
    g.newton_krylov_step(s["U"], case["cfl"], krylov_dim=case["krylov_dim"], precond=case["precond"])
    # the snapshot a user stores: the step's finite-difference products (and its
    # FP32 Krylov basis) turn the last bit of a residual into 1e-9 to 1e-7 of
    # the state, so its FP64 digits beyond single precision carry nothing
    return dict(U=s["U"].float())


def work(case):
    """Inputs read once, outputs written once; operations of the method per cell:
    three Rusanov fluxes, 27 limited slopes, recovery and gather about 1100 for
    a residual, about 2600 for its reverse."""
    cells = sum(a * b * c for a, b, c in _shapes(case))
    size = 8 if case["precision"] == "fp64" else 4
    kind = case["kind"]
    state = 9 * cells * size
    if kind in ("residual", "ensemble"):
        return dict(bytes=2 * state, flops=1100 * cells)
    if kind == "gradient":
        return dict(bytes=4 * state, flops=3700 * cells)
    if kind == "pseudo_time":
        return dict(bytes=2 * 72 * cells, flops=1150 * cells * case["steps"])
    if kind == "newton_krylov":   # about half the Krylov space, two residuals per product
        return dict(bytes=2 * 72 * cells, flops=1100 * cells * case["krylov_dim"])
    return dict(bytes=3 * 72 * cells, flops=2600 * cells * case["krylov_dim"] * case["passes"] / 4)


# ---------------------------------------------------------------------------
# the operator in plain float64 torch operations
# ---------------------------------------------------------------------------
def _geometry(shape):
    nr, nt, np_ = shape
    rf = _t(ci.radial_faces(nr))
    rc = 0.5 * (rf[:-1] + rf[1:])
    dth, dph = math.pi / nt, 2.0 * math.pi / np_
    half = 2.0 * math.sin(0.5 * dph)
    tl = dth * torch.arange(nt, dtype=F64, device=DEV)
    tc, pc = tl + 0.5 * dth, dph * (torch.arange(np_, dtype=F64, device=DEV) + 0.5)
    cp, sp = torch.cos(pc), torch.sin(pc)
    # area vectors: integrals of the unit normal over the faces
    X = 0.5 * (dth - torch.cos(2 * tl + dth) * math.sin(dth))
    Z = 0.5 * torch.sin(2 * tl + dth) * math.sin(dth)
    o = torch.ones_like(cp)
    Sr = torch.stack([X[:, None] * half * cp, X[:, None] * half * sp, Z[:, None] * dph * o])
    tf = tl[1:]
    St = torch.stack([(torch.sin(tf) * torch.cos(tf))[:, None] * half * cp,
                      (torch.sin(tf) * torch.cos(tf))[:, None] * half * sp,
                      -(torch.sin(tf) ** 2)[:, None] * dph * o])
    pf = pc - 0.5 * dph
    Sp = torch.stack([-torch.sin(pf), torch.cos(pf), torch.zeros_like(pf)]) * dth
    rb = 0.5 * (rf[1:] ** 2 - rf[:-1] ** 2)
    vol = ((rf[1:] ** 3 - rf[:-1] ** 3) / 3.0)[:, None] * (torch.cos(tl) - torch.cos(tl + dth)) * dph
    st, ct = torch.sin(tc), torch.cos(tc)
    rhat = torch.stack([st[:, None] * cp, st[:, None] * sp, ct[:, None] * o])
    return dict(rf=rf, rc=rc, Sr=Sr, St=St, Sp=Sp, rb=rb, vol=vol[:, :, None], rhat=rhat)


def _limited(a, b, limiter):
    if limiter == "minmod":
        return torch.where(a * b > 0, torch.where(a.abs() < b.abs(), a, b), torch.zeros_like(a))
    e = 1e-12
    return (a * (b * b + e) + b * (a * a + e)) / (a * a + b * b + 2 * e)


def _dot(a, b):
    return a[0] * b[0] + a[1] * b[1] + a[2] * b[2]


def _flux(L, R, S):
    """Rusanov + GLM flux of the primitive states through the area vectors S; and its speed x area."""
    A = torch.sqrt(_dot(S, S))
    n = S / A

    def side(w):
        rho, v, b, p, psi = w[0], w[1:4], w[4:7], w[7], w[8]
        un, bn, b2 = _dot(v, n), _dot(b, n), _dot(b, b)
        en = p / (ci.GAMMA - 1.0) + 0.5 * rho * _dot(v, v) + 0.5 * b2
        a2 = ci.GAMMA * p / rho
        s = a2 + b2 / rho
        cf = torch.sqrt(0.5 * (s + torch.sqrt(torch.clamp(s * s - 4 * a2 * bn * bn / rho, min=0.0))))
        pt = p + 0.5 * b2
        F = torch.cat([(rho * un)[None], rho * un * v + pt * n - bn * b, un * b - bn * v + psi * n,
                       ((en + pt) * un - bn * _dot(v, b))[None], bn[None]])
        Uc = torch.cat([rho[None], rho * v, b, en[None], psi[None]])
        return F, Uc, un.abs() + cf

    FL, UL, sL = side(L)
    FR, UR, sR = side(R)
    lam = torch.clamp(torch.maximum(sL, sR), min=1.0)
    return (0.5 * (FL + FR) - 0.5 * lam * (UR - UL)) * A, lam * A


def _exact_residual(U, Br, case):
    shape = tuple(U.shape[1:])
    nr, nt, np_ = shape
    g = _geometry(shape)
    rho, V, B, E, psi = U[0], U[1:4] / U[0], U[4:7], U[7], U[8]
    p = (ci.GAMMA - 1.0) * (E - 0.5 * rho * _dot(V, V) - 0.5 * _dot(B, B))
    W = torch.cat([rho[None], V, B, p[None], psi[None]])
    e = g["rhat"]
    # inner ghost: B_r prescribed, E_b = 0
    w = W[:, 0]
    vi, bi = w[1:4], w[4:7]
    Bb = Br * e + (bi - _dot(bi, e) * e)
    s = (VR_STAR * Br if case["inner_bc"] == "low_e_wp" else _dot(vi, Bb)) / _dot(Bb, Bb)
    one = torch.ones_like(w[:1])
    gin = torch.cat([one, 2 * s * Bb - vi, 2 * Bb - bi, ci.parker_sound_speed2() * one, -w[8:9]])
    # outer ghost: rho, p and B_r ~ r^-2, psi_b = 0
    w = W[:, -1]
    rI = g["rc"][-1]
    f = (rI / (2.0 * g["rf"][-1] - rI)) ** 2
    gout = torch.cat([w[:1] * f, w[1:4], w[4:7] + (f - 1.0) * _dot(w[4:7], e) * e, w[7:8] * f, -w[8:9]])
    acc = torch.zeros_like(U)
    # r faces
    rc, rf = g["rc"], g["rf"]
    c = torch.cat([(2 * rf[0] - rc[0])[None], rc, (2 * rf[-1] - rc[-1])[None]])
    x = torch.cat([gin[:, None], W, gout[:, None]], 1)
    d = (x[:, 1:] - x[:, :-1]) / (c[1:] - c[:-1])[:, None, None]
    sl = _limited(d[:, :-1], d[:, 1:], case["limiter"])
    up = W + sl * (rf[1:] - rc)[:, None, None]
    lo = W - sl * (rc - rf[:-1])[:, None, None]
    L = torch.cat([gin[:, None], up[:, :-1], W[:, -1:]], 1)
    R = torch.cat([W[:, :1], lo[:, 1:], gout[:, None]], 1)
    F, lr = _flux(L, R, g["Sr"][:, None] * (rf ** 2)[:, None, None])
    acc = acc + F[:, :-1] - F[:, 1:]
    lam = lr[:-1] + lr[1:]
    # theta faces (the pole faces have no area)
    x = torch.cat([W[:, :, :1].roll(np_ // 2, 3), W, W[:, :, -1:].roll(np_ // 2, 3)], 2)
    d = x[:, :, 1:] - x[:, :, :-1]
    sl = 0.5 * _limited(d[:, :, :-1], d[:, :, 1:], case["limiter"])
    F, lt = _flux((W + sl)[:, :, :-1], (W - sl)[:, :, 1:], g["St"][:, None, :nt - 1] * g["rb"][:, None, None])
    z = torch.zeros_like(F[:, :, :1])
    acc = acc + torch.cat([z, F], 2) - torch.cat([F, z], 2)
    lam = lam + torch.cat([z[0], lt], 1) + torch.cat([lt, z[0]], 1)
    # phi faces
    d = W - W.roll(1, 3)
    sl = 0.5 * _limited(d, d.roll(-1, 3), case["limiter"])
    F, lp = _flux((W + sl).roll(1, 3), W - sl, (g["Sp"][:, None, None, :] * g["rb"][:, None, None]).expand(3, *shape))
    acc = acc + F - F.roll(-1, 3)
    lam = lam + lp + lp.roll(-1, 2)
    # sources
    R = acc / g["vol"]
    gv = -(ci.G0_SOLAR / rc ** 2)[:, None, None] * e[:, None]
    src = torch.cat([torch.zeros_like(R[:1]), W[0] * gv, torch.zeros_like(R[:3]), (W[0] * _dot(V, gv))[None],
                     torch.zeros_like(R[:1])])
    return R + src, (g["vol"] / lam).min()


def exact(case, seed):
    kind = case["kind"]
    if kind in ("newton_krylov", "adjoint"):
        return None
    data = _inputs(case, seed)
    if kind == "ensemble":
        return dict(R=[_exact_residual(U.double(), Br, case)[0] for _, U, Br in data])
    _, U, Br = data[0]
    if kind == "residual":
        R, dtmin = _exact_residual(U.double(), Br, case)
        if case["precision"] == "fp32":
            return dict(R=R)
        return dict(R=R, norms=torch.sqrt((R * R).sum((1, 2, 3))), dtmin=dtmin.reshape(1))
    if kind == "gradient":
        gen = torch.Generator(device=DEV).manual_seed(seed + 4)
        Rbar = torch.randn(U.shape, dtype=F64, device=DEV, generator=gen).to(U.dtype).double()
        Ux, Bx = U.double().requires_grad_(True), Br.requires_grad_(True)
        R = _exact_residual(Ux, Bx, case)[0]
        Ubar, Brbar = torch.autograd.grad(R, (Ux, Bx), Rbar)
        out = dict(R=R.detach(), Ubar=Ubar)
        return dict(out, Brbar=Brbar) if case["precision"] == "fp64" else out
    for _ in range(case["steps"]):
        R, dtmin = _exact_residual(U, Br, case)
        U = U + case["cfl"] * dtmin * R
    return dict(U=U)
