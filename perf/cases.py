"""The calls by which the solver's speed is judged, over the range of sizes, orders and options it is used with.

Kinds of case, each one pass through the public binding (jfnk.Context, jfnk.Batch):

  residual   f = M^-1 L_h(U'), the explicit operator (explicit steppers, diagnostics, every Newton residual)
  jv         one Jacobian-free product with a given step eps
  precond    one application of the FP32 DG->FV multigrid preconditioner, linearisation included
  step       one implicit step (backward Euler or SDIRK2), what a forecast program calls in its loop
  ensemble   one batched step of several uneven members on their own streams

The states are those of the repository's test cases (a warm or cold potential-temperature bubble, an
inertia-gravity wave), the bubble drawn and the noise made from the seed.  Contexts (tables, workspace, captured
graphs) are made once in prepare(), as a forecast program keeps them; a step starts from a fixed state U0 that is
copied into the work vector, so that every pass does the same work.  Steps are solved to a Newton tolerance of 1e-9
(the library's default is 1e-8): what they return is determined by that tolerance, and by nothing more.
"""
import math

import numpy as np
import torch

import paper_2505_24504_gb300 as P
from paper_2505_24504_gb300 import presets

PHYS = {   # constants of the rising-bubble / inertia-gravity and of the density-current test cases
    "robert": dict(cp=1005.0, cv=717.95, g=9.80665, p0=1.0e5),
    "straka": dict(cp=1004.0, cv=717.0, g=9.81, p0=1.0e5),
}
DOMAIN = {"bubble": (20000.0, 10000.0), "current": (51200.0, 6400.0), "wave": (300000.0, 10000.0)}
DEV = "cuda"
ADT = 1.0 - math.sqrt(2.0) / 2.0    # SDIRK2's alpha: alpha dt is what a stage passes to products and preconditioner


def _case(kind, scene, nx, nz, k, name=None, **kw):
    c = {"kind": kind, "scene": scene, "nx": nx, "nz": nz, "k": k, **kw}
    return c if name is None else {"name": name, **c}


def listed():
    return [
        # the smallest grid of the test cases (7,200 unknowns): two short launches, latency
        _case("residual", "bubble", 20, 10, 2, name="residual_q2_20x10"),
        # the density current's full grid, viscous: interior-penalty terms on every face
        _case("residual", "current", 256, 32, 2, name="residual_visc_q2_256x32"),
        # the largest member of the uneven ensemble (5.12 M unknowns)
        _case("residual", "bubble", 320, 160, 4, name="residual_q4_320x160"),
        # the Krylov product of the 819,200-unknown warm bubble, eps as the full-size parity test gives it
        _case("jv", "bubble", 160, 80, 3, name="jv_q3_160x80", eps=1e-3),
        # an odd, ragged viscous grid of lowest order
        _case("jv", "current", 201, 37, 1, name="jv_visc_q1_201x37", eps=1e-3),
        # preconditioner of the inertia-gravity wave: periodic, three element rows, launch latency
        _case("precond", "wave", 80, 3, 3, name="precond_q3_80x3", levels=3, key="mg111111V"),
        # ... and of the 819,200-unknown warm bubble with its recorded schedule
        _case("precond", "bubble", 160, 80, 3, name="precond_q3_160x80", levels=5, preset="WARM_BUBBLE_Q3_160x80"),
        # one backward-Euler step with the library's default options (FP64 preconditioner, three levels)
        _case("step", "bubble", 20, 10, 2, name="step_be_q2_20x10", levels=3, key="mg111111V", prec=64, scheme=0,
              cfl=10.0),
        # the inertia-gravity wave at its test-case step
        _case("step", "wave", 80, 3, 3, name="step_q3_80x3", levels=3, key="mg111111V", prec=32, scheme=1, dt=25.0),
        # the viscous density current at its test-case step
        _case("step", "current", 256, 32, 2, name="step_visc_q2_256x32", levels=4, key="mg111111V", prec=32, scheme=1,
              dt=1.0),
        # the warm bubble of the benchmark: SDIRK2 at 20x the acoustic CFL step
        _case("step", "bubble", 160, 80, 3, name="step_q3_160x80", levels=5, preset="WARM_BUBBLE_Q3_160x80", prec=32,
              scheme=1, cfl=20.0),
        # eight members, orders 1..4 on 40x20 and 80x40 quads, stepped together
        _case("ensemble", "bubble", 40, 20, 1, name="ensemble_8", members=8, levels=3, key="mg111111V", prec=32,
              scheme=1, cfl=10.0),
    ]


def _grid(rng, k, most, least=512.0):
    """A grid whose unknowns are spread over the logarithm of [least, most], odd counts among them."""
    n = math.exp(rng.uniform(math.log(least), math.log(most)))
    el = max(2.0, n / (4 * (k + 1) ** 2))
    aspect = math.exp(rng.uniform(0.0, math.log(8.0)))
    nx = max(2, min(400, int(math.sqrt(el * aspect))))
    return nx, max(2, min(200, int(el / nx)))


def draw(rng):
    kind = rng.choice(["residual", "residual", "jv", "precond", "step"])
    scene = rng.choice(["bubble", "bubble", "current", "wave"])
    k = rng.choice([1, 2, 3, 4])
    if kind == "residual":
        return _case(kind, scene, *_grid(rng, k, 4.0e6), k)
    if kind == "jv":
        return _case(kind, scene, *_grid(rng, k, 8.0e5), k, eps=rng.choice([1e-3, 1e-2]))
    levels = rng.choice([2, 3, 4])
    key = rng.choice(["mg111111V", "mg111111W", "mg131211V"])
    if kind == "precond":
        return _case(kind, scene, *_grid(rng, k, 8.0e5), k, levels=levels, key=key)
    return _case(kind, scene, *_grid(rng, k, 1.0e5, least=4000.0), k, levels=levels, key="mg111111V",
                 prec=rng.choice([32, 32, 64]), scheme=rng.choice([0, 1]), cfl=rng.choice([5.0, 10.0]))


# ---- set-up ---------------------------------------------------------------
def _physics(case):
    s = case["scene"]
    c = PHYS["straka" if s == "current" else "robert"]
    return dict(c, theta0=250.0 if s == "wave" else 300.0, mu=75.0 if s == "current" else 0.0,
                background=2 if s == "wave" else 0, ubg=20.0 if s == "wave" else 0.0, N_bv=0.01)


def _dt(case, k=None, nx=None, nz=None):
    if "dt" in case:
        return case["dt"]
    k, nx, nz = k or case["k"], nx or case["nx"], nz or case["nz"]
    ph, (lx, lz) = _physics(case), DOMAIN[case["scene"]]
    c = math.sqrt(ph["cp"] / ph["cv"] * (ph["cp"] - ph["cv"]) * ph["theta0"])
    return case.get("cfl", 10.0) * min(lx / nx, lz / nz) / ((2 * k + 1) * c)


def _context(case, k=None, nx=None, nz=None):
    k, nx, nz = k or case["k"], nx or case["nx"], nz or case["nz"]
    ph, (lx, lz) = _physics(case), DOMAIN[case["scene"]]
    grid = P.Grid(nx, nz, 0.0, lx, 0.0, lz, int(case["scene"] == "wave"))
    phys = P.Physics(ph["cp"], ph["cv"], ph["g"], ph["p0"], ph["theta0"], ph["mu"], ph["background"], ph["ubg"], 0.0,
                     ph["N_bv"])
    opt = dict(fv_levels=case.get("levels", 3), precond_prec=case.get("prec", 32), newton_tol=1e-9)
    opt.update(getattr(presets, case["preset"]) if "preset" in case else dict(mg_key=case.get("key", "mg111111V")))
    return P.Context(grid, k, phys, P.Opts.defaults(**opt))


def _initial(ctx, case, seed):
    """The scene's potential-temperature perturbation, drawn from the seed, inserted by the library."""
    r = np.random.Generator(np.random.Philox(seed))
    x, z = (torch.from_numpy(a).to(DEV) for a in ctx.node_coords())
    lx, lz = DOMAIN[case["scene"]]
    if case["scene"] == "wave":
        th = r.uniform(0.2, 1.0) * torch.sin(math.pi * z / lz) / (1.0 + ((x - r.uniform(0.25, 0.75) * lx) / 5000.0) ** 2)
    else:
        cold = case["scene"] == "current"
        amp, xc = (r.uniform(-15.0, -5.0), 0.0) if cold else (r.uniform(1.0, 4.0), r.uniform(6000.0, 14000.0))
        zc = r.uniform(2500.0, 3500.0) if cold else r.uniform(1500.0, 3000.0)
        d = torch.sqrt(((x - xc) / (4000.0 if cold else 2000.0)) ** 2 + ((z - zc) / 2000.0) ** 2)
        th = torch.where(d < 1.0, 0.5 * amp * (1.0 + torch.cos(math.pi * d)), torch.zeros_like(d))
        g = torch.Generator(device=DEV).manual_seed(int(seed))
        th = th + 0.1 * (2.0 * torch.rand(th.shape, dtype=torch.float64, device=DEV, generator=g) - 1.0)
    U = torch.empty(ctx.N, dtype=torch.float64, device=DEV)
    ctx.jfnk_init_state(th, U)
    return U


def _perturbation(n, seed):
    """A random state of the magnitudes that occur some steps into a run."""
    g = torch.Generator(device=DEV).manual_seed(int(seed) + 7919)
    y = torch.randn(4, n // 4, dtype=torch.float64, device=DEV, generator=g)
    return (y * torch.tensor([1e-3, 1.0, 1.0, 0.3], dtype=torch.float64, device=DEV)[:, None]).reshape(-1)


def prepare(case, seed):
    kind = case["kind"]
    s = {"case": case}
    if kind == "ensemble":
        ctxs, U0, dts = [], [], []
        for m in range(case["members"]):
            k, f = 1 + m % 4, 1 + (m // 4) % 2
            ctxs.append(_context(case, k, f * case["nx"], f * case["nz"]))
            U0.append(_initial(ctxs[-1], case, seed + 1000 * (m + 1)))
            dts.append(_dt(case, k, f * case["nx"], f * case["nz"]))
        return dict(s, batch=P.Batch(ctxs), U0=U0, U=[u.clone() for u in U0], dts=dts,
                    schemes=[case["scheme"]] * len(ctxs))
    ctx = _context(case)
    U = _initial(ctx, case, seed)
    s.update(ctx=ctx, U0=U, U=U.clone())
    if kind != "step":
        s["U0"] = U + _perturbation(ctx.N, seed)
        s["out"] = torch.empty_like(U)
    if kind == "jv":
        s["fU"], s["y"] = torch.empty_like(U), _perturbation(ctx.N, seed + 1)
        ctx.dg_residual(s["U0"], s["fU"])
    if kind == "precond":
        s["y"] = _perturbation(ctx.N, seed + 1)
    return s


def run(s):
    case, kind = s["case"], s["case"]["kind"]
    if kind == "residual":
        s["ctx"].dg_residual(s["U0"], s["out"])
        return s["out"]
    if kind == "jv":
        s["ctx"].jv_product(s["U0"], s["fU"], s["y"], ADT * _dt(case), case["eps"], s["out"])
        return s["out"]
    if kind == "precond":
        # computed in FP32 and widened: handed on as the FP32 values it holds
        s["ctx"].mg_precondition(s["U0"], ADT * _dt(case), s["y"], s["out"])
        return s["out"].float()
    if kind == "step":
        s["U"].copy_(s["U0"])
        s["ctx"].implicit_step(s["U"], _dt(case), scheme=case["scheme"])
        return s["U"]
    for u, u0 in zip(s["U"], s["U0"]):
        u.copy_(u0)
    torch.cuda.current_stream().synchronize()   # the members run on streams of their own
    s["batch"].jfnk_batch_step(s["U"], s["dts"], s["schemes"])
    return s["U"]


# ---- what a pass cannot do without ----------------------------------------
def work(case):
    if case["kind"] == "ensemble":
        w = [work(dict(case, kind="step", k=1 + m % 4, nx=(1 + (m // 4) % 2) * case["nx"],
                       nz=(1 + (m // 4) % 2) * case["nz"])) for m in range(case["members"])]
        return {q: sum(x[q] for x in w) for q in ("bytes", "flops")}
    nx, nz, n1 = case["nx"], case["nz"], case["k"] + 1
    nodes, faces = nx * nz * n1 * n1, (nz * (nx + 1) + nx * (nz + 1)) * n1
    N, visc = 4 * nodes, case["scene"] == "current"
    # Euler: HLLC and traces per face point, fluxes, derivatives and lifts per node; viscous: gradients, SIPG terms
    op = faces * (70 + 16 * n1 + (60 + 16 * n1 if visc else 0)) + nodes * (60 + 16 * n1 + (24 + 16 * n1 if visc else 0))
    pre = 3 * op + 4 * nodes * 500          # three DG products and about four fine-grid FV products
    if case["kind"] == "residual":
        return {"bytes": 16 * N, "flops": op}
    if case["kind"] == "jv":
        return {"bytes": 32 * N, "flops": op + 6 * N}
    if case["kind"] == "precond":
        return {"bytes": 24 * N, "flops": op + pre}
    # a step: typically 4 Newton iterations a stage with 7 Krylov vectors each, every basis vector kept in memory
    newton = 4 * (2 if case["scheme"] else 1)
    return {"bytes": newton * 7 * (32 + 16 * 7) * N, "flops": newton * (op + 7 * (op + pre + 4 * 4 * N))}


# ---- the same values from plain torch in 64 bits ---------------------------
def _lagrange(nodes, x):
    return np.array([[np.prod([(xx - b) / (a - b) for b in nodes if b != a]) for a in nodes] for xx in x])


def _lagrange_deriv(nodes, x):
    def d(a, xx):
        rest = [b for b in nodes if b != a]
        return sum(np.prod([1.0 / (a - m)] + [(xx - b) / (a - b) for b in rest if b != m]) for m in rest)
    return np.array([[d(a, xx) for a in nodes] for xx in x])


class _Plain:
    """The DG operator, its FV levels and the multigrid cycle, written out in torch (float64, and complex128 for
    derivatives by a complex step)."""

    def __init__(self, case):
        self.nx, self.nz, self.n1 = case["nx"], case["nz"], case["k"] + 1
        self.ph, (self.lx, self.lz) = _physics(case), DOMAIN[case["scene"]]
        self.R = self.ph["cp"] - self.ph["cv"]
        self.gam = self.ph["cp"] / self.ph["cv"]
        self.per = case["scene"] == "wave"
        self.hx, self.hz = self.lx / self.nx, self.lz / self.nz
        xi, w = np.polynomial.legendre.leggauss(self.n1)
        t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(DEV)  # noqa: E731
        self.xi, self.w, self.D = xi, t(w), t(_lagrange_deriv(xi, xi))
        self.l = [t(_lagrange(xi, [e])[0]) for e in (-1.0, 1.0)]
        self.dl = [t(_lagrange_deriv(xi, [e])[0]) for e in (-1.0, 1.0)]
        zr = (np.arange(self.nz)[:, None] + 0.5 * (1.0 + xi[None, :])) * self.hz
        self.ubv, self.dubv = self.background(zr)                                  # (4, nz, b)
        self.ubh, self.dubh = self.background(np.arange(self.nz + 1) * self.hz)    # (4, nz+1)
        cen = np.array([-1.0 + (2 * i + 1) / self.n1 for i in range(self.n1)])
        V = _lagrange(xi, cen)
        self.V, self.Vi = t(V), t(np.linalg.inv(V))

    def background(self, z):
        ph, R = self.ph, self.R
        if ph["background"] == 0:
            T = ph["theta0"] - ph["g"] * z / ph["cp"]
            p = ph["p0"] * (T / ph["theta0"]) ** (ph["cp"] / R)
            th, dT, dth = np.full_like(T, ph["theta0"]), np.full_like(T, -ph["g"] / ph["cp"]), np.zeros_like(T)
        else:
            H = ph["g"] / ph["N_bv"] ** 2
            al, e = ph["g"] * H / (ph["cp"] * ph["theta0"]), np.exp(z / H)
            th, T = ph["theta0"] * e, ph["theta0"] * (al - (al - 1.0) * e)
            p = ph["p0"] * np.exp(ph["cp"] / R * (np.log(T / ph["theta0"]) - z / H))
            dT, dth = -ph["theta0"] * (al - 1.0) * e / H, th / H
        rho = p / (R * T)
        drho = (-rho * ph["g"] * T - p * dT) / (R * T * T)
        u, o = ph["ubg"], np.zeros_like(rho)
        return (torch.from_numpy(np.stack([rho, u * rho, o, rho * th])).to(DEV),
                torch.from_numpy(np.stack([drho, u * drho, o, drho * th + rho * dth])).to(DEV))

    def pressure(self, E):
        return self.ph["p0"] * (self.R * E / self.ph["p0"]) ** self.gam

    def flux(self, U, d):
        un = U[1 + d] / U[0]
        F = [U[1 + d], U[1] * un, U[2] * un, U[3] * un]
        F[1 + d] = F[1 + d] + self.pressure(U[3])
        return torch.stack(F)

    def hllc(self, L, Rr, d):
        n, t = 1 + d, 2 - d
        re = lambda a: a.real if a.is_complex() else a  # noqa: E731
        uL, uR = L[n] / L[0], Rr[n] / Rr[0]
        pL, pR = self.pressure(L[3]), self.pressure(Rr[3])
        cL, cR = torch.sqrt(self.gam * pL / L[0]), torch.sqrt(self.gam * pR / Rr[0])
        SL = torch.where(re(uL - cL) <= re(uR - cR), uL - cL, uR - cR)
        SR = torch.where(re(uL + cL) >= re(uR + cR), uL + cL, uR + cR)
        mL, mR = L[0] * (SL - uL), Rr[0] * (SR - uR)
        S = (pR - pL + uL * mL - uR * mR) / (mL - mR)

        def star(U, un, Sk):
            f = U[0] * (Sk - un) / (Sk - S)
            q = [f, None, None, f * (U[3] / U[0])]
            q[n], q[t] = f * S, f * (U[t] / U[0])
            return self.flux(U, d) + Sk * (torch.stack(q) - U)
        out = torch.where(re(SR) >= 0, star(Rr, uR, SR), self.flux(Rr, d))
        out = torch.where(re(S) >= 0, star(L, uL, SL), out)
        return torch.where(re(SL) >= 0, self.flux(L, d), out)

    def face(self, L, Rr, d):
        """Flux through one face layer; None on a side: a slip wall there."""
        m = lambda A: torch.stack([-a if i == 1 + d else a for i, a in enumerate(A)])  # noqa: E731
        return self.hllc(m(Rr) if L is None else L, m(L) if Rr is None else Rr, d)

    def faces(self, lo, hi, ub, d, axis):
        """Perturbation fluxes of all faces along `axis`: lo / hi the traces at an element's lower / upper end
        (perturbations), ub the background at every face (broadcastable)."""
        n = lo.shape[axis]
        at = lambda A, a, b: A.narrow(axis, a, b - a)  # noqa: E731
        bg = lambda a, b: ub if ub.shape[axis] == 1 else at(ub, a, b)  # noqa: E731
        H = lambda l, r, b: (self.face(None if l is None else l + b, None if r is None else r + b, d)  # noqa: E731
                             - self.face(None if l is None else b + 0 * l, None if r is None else b + 0 * r, d))
        inner = H(at(hi, 0, n - 1), at(lo, 1, n), bg(1, n)) if n > 1 else None
        if d == 0 and self.per:
            first = last = H(at(hi, n - 1, n), at(lo, 0, 1), bg(0, 1))
        else:
            first, last = H(None, at(lo, 0, 1), bg(0, 1)), H(at(hi, n - 1, n), None, bg(n, n + 1))
        return torch.cat([first] + ([inner] if n > 1 else []) + [last], dim=axis)

    def visc(self, U, dU):
        return self.ph["mu"] * torch.stack([torch.zeros_like(dU[0] * U[0])] + [dU[i] - U[i] / U[0] * dU[0] for i in (1, 2, 3)])

    def rhs(self, Up):
        """f = M^-1 L_h(U'), arrays (4, nz, nx, b, a)."""
        ein = lambda s, A, B: torch.einsum(s, A.to(B.dtype), B)  # noqa: E731
        w, D, (lm, lp), (dlm, dlp) = self.w, self.D, self.l, self.dl
        hx, hz, mu = self.hx, self.hz, self.ph["mu"]
        ub = self.ubv[:, :, None, :, None]
        U = Up + ub
        b0 = ub + 0 * Up.real if Up.is_complex() else ub + 0 * Up
        Gx, Gz = self.flux(U, 0) - self.flux(b0, 0), self.flux(U, 1) - self.flux(b0, 1)
        if mu:
            Gx = Gx - self.visc(U, 2.0 / hx * ein("qa,vzxba->vzxbq", D, Up))
            Gz = Gz - self.visc(U, 2.0 / hz * ein("br,vzxra->vzxba", D, Up) + self.dubv[:, :, None, :, None])
        wD = w[:, None] * D
        f = 2.0 / hx * ein("qa,vzxbq->vzxba", wD, Gx) / w + 2.0 / hz * ein("rb,vzxra->vzxba", wD, Gz) / w[:, None]
        f[2] -= self.ph["g"] * Up[0]
        for d, h, sub, axis in ((0, hx, "a,vzxba->vzxb", 2), (1, hz, "b,vzxba->vzxa", 1)):
            lo, hi = ein(sub, lm, Up), ein(sub, lp, Up)
            ubf = self.ubv[:, :, None, :] if d == 0 else self.ubh[:, :, None, None]
            H = self.faces(lo, hi, ubf, d, axis)
            n = lo.shape[axis]
            up = (lambda A: A[..., None]) if d == 0 else (lambda A: A[..., None, :])
            vec = (lambda v: v) if d == 0 else (lambda v: v[:, None])
            sc = 2.0 / h / vec(w)
            f = f + sc * (vec(lm) * up(H.narrow(axis, 0, n)) - vec(lp) * up(H.narrow(axis, 1, n)))
            if not mu:
                continue
            glo, ghi = 2.0 / h * ein(sub, dlm, Up), 2.0 / h * ein(sub, dlp, Up)
            iL, iR = list(range(n - 1)), list(range(1, n))
            if d == 0 and self.per:
                iL, iR = iL + [n - 1], iR + [0]
            if not iL:
                continue
            a, b = torch.tensor(iL, device=DEV), torch.tensor(iR, device=DEV)
            L, Rr = hi.index_select(axis, a), lo.index_select(axis, b)
            ubi = ubf if d == 0 else ubf.index_select(1, b)
            dub = 0.0 if d == 0 else self.dubh[:, :, None, None].index_select(1, b)
            J = L - Rr
            sL, sR = 0.5 * self.visc(L + ubi, J), 0.5 * self.visc(Rr + ubi, J)
            avg = 0.5 * (self.visc(L + ubi, ghi.index_select(axis, a) + dub) + self.visc(Rr + ubi, glo.index_select(axis, b) + dub))
            pen = 2.0 * self.n1 ** 2 / h * (sL + sR)
            f.index_add_(axis, a, sc * (vec(lp) * up(avg - pen) + 2.0 / h * vec(dlp) * up(sL)))
            f.index_add_(axis, b, sc * (vec(lm) * up(pen - avg) + 2.0 / h * vec(dlm) * up(sR)))
        return f

    # -- the FV levels and the cycle --
    def fv_rhs(self, lev, up):
        NX, NZ, Hx, Hz, ub = lev
        U = up + ub
        Fx = self.faces(up, up, ub, 0, 2)
        b = ub + 0 * (up.real if up.is_complex() else up)
        Fz = [self.face(None, U[:, :1], 1) - self.face(None, b[:, :1], 1)]
        if NZ > 1:
            Fz.append(self.hllc(U[:, :-1], U[:, 1:], 1) - self.hllc(b[:, :-1], b[:, 1:], 1))
        Fz.append(self.face(U[:, -1:], None, 1) - self.face(b[:, -1:], None, 1))
        Fz = torch.cat(Fz, dim=1)
        f = -((Fx[:, :, 1:] - Fx[:, :, :-1]) / Hx + (Fz[:, 1:] - Fz[:, :-1]) / Hz)
        f[2] -= self.ph["g"] * up[0]
        if self.ph["mu"]:
            phi = U[1:] / U[0]
            Z = lambda A: torch.zeros_like(A)  # noqa: E731
            v = lambda r0, r1, p0, p1, h: self.ph["mu"] * 0.5 * (r0 + r1) * (p1 - p0) / h  # noqa: E731
            ix = v(U[0][:, :-1], U[0][:, 1:], phi[:, :, :-1], phi[:, :, 1:], Hx)
            ends = v(U[0][:, -1:], U[0][:, :1], phi[:, :, -1:], phi[:, :, :1], Hx) if self.per else Z(phi[:, :, :1])
            ix = torch.cat([ends, ix, ends], dim=2)
            iz = v(U[0][:-1], U[0][1:], phi[:, :-1], phi[:, 1:], Hz)
            iz = torch.cat([Z(phi[:, :1]), iz, Z(phi[:, :1])], dim=1)
            f[1:] += (ix[:, :, 1:] - ix[:, :, :-1]) / Hx + (iz[:, 1:] - iz[:, :-1]) / Hz
        return f

    def mass(self, u, v, to_dg):
        """Mean of the DG polynomial minus the mean of its subcell values, per element."""
        m = torch.einsum("b,a,vzxba->vzx", self.w, self.w, u) / 4.0 - v.mean(dim=(3, 4))
        return m[..., None, None] if to_dg else -m[..., None, None]

    def to_fv(self, u):
        v = torch.einsum("jb,ia,vzxba->vzxji", self.V, self.V, u)
        v = v - self.mass(u, v, False)
        return v.permute(0, 1, 3, 2, 4).reshape(4, self.nz * self.n1, self.nx * self.n1)

    def to_dg(self, v):
        v = v.reshape(4, self.nz, self.n1, self.nx, self.n1).permute(0, 1, 3, 2, 4)
        u = torch.einsum("bj,ai,vzxji->vzxba", self.Vi, self.Vi, v)
        return u - self.mass(u, v, True)

    def precondition(self, U, adt, r, key, levels, s_fv, s_dg):
        n1 = self.n1
        a, b, c, d, e, f = (int(q) for q in key[2:8])
        cycles = 1 if key[8] == "V" else 2
        sizes, facs = [(self.nx * n1, self.nz * n1)], []
        steps = [2] * int(math.log2(n1)) if n1 & (n1 - 1) == 0 else [n1]
        while len(sizes) < levels:
            fac = steps.pop(0) if steps else 2
            X, Z = sizes[-1]
            if X % fac or Z % fac or X < 2 or Z < 2:
                break
            sizes.append((X // fac, Z // fac))
            facs.append(fac)
        shape = (4, self.nz, self.nx, n1, n1)
        U, r = U.reshape(shape), r.reshape(shape)
        h = 1e-20
        jac = lambda F, u, x: x - adt * F(torch.complex(u, h * x)).imag / h  # noqa: E731
        speed = lambda A: torch.sqrt(self.gam * self.pressure(A[3]) / A[0])  # noqa: E731
        lev, us, dts = [], [], []
        for q, (X, Z) in enumerate(sizes):
            Hx, Hz = self.lx / X, self.lz / Z
            ub = self.background((np.arange(Z) + 0.5) * Hz)[0][:, :, None]
            lev.append((X, Z, Hx, Hz, ub))
            u = self.to_fv(U) if q == 0 else us[-1].reshape(4, Z, facs[q - 1], X, facs[q - 1]).mean(dim=(2, 4))
            us.append(u)
            A = u + ub
            cs = speed(A)
            sx, sz = (A[1] / A[0]).abs() + cs, (A[2] / A[0]).abs() + cs
            px = torch.cat([sx[:, -1:] if self.per else sx[:, :1], sx, sx[:, :1] if self.per else sx[:, -1:]], dim=1)
            pz = torch.cat([sz[:1], sz, sz[-1:]], dim=0)
            ex, ez = torch.maximum(px[:, :-1], px[:, 1:]), torch.maximum(pz[:-1], pz[1:])
            lam = 0.5 * (ex[:, :-1] + ex[:, 1:]) / Hx + 0.5 * (ez[:-1] + ez[1:]) / Hz + 2 * self.ph["mu"] * (Hx ** -2 + Hz ** -2)
            dts.append(s_fv / (1.0 + adt * lam))
        A = U + self.ubv[:, :, None, :, None]
        vm = (torch.sqrt((A[1] / A[0]) ** 2 + (A[2] / A[0]) ** 2) + speed(A)).amax(dim=(2, 3))
        lam = n1 ** 2 * vm * (1 / self.hx + 1 / self.hz) + 2 * self.ph["mu"] * n1 ** 4 * (self.hx ** -2 + self.hz ** -2)
        dtd = (s_dg / (1.0 + adt * lam))[None, :, :, None, None]

        def smooth(x, rhs, dt, J, n):
            for _ in range(n):
                x = dt * rhs if x is None else x + dt * (rhs - J(x))
            return x

        def mg(q, x, rhs):
            J = lambda y: jac(lambda s: self.fv_rhs(lev[q], s), us[q], y)  # noqa: E731
            x = smooth(x, rhs, dts[q], J, c if q == 0 else e)
            if q + 1 < len(lev):
                res = -rhs if x is None else J(x) - rhs
                X, Z, fac, v = lev[q + 1][0], lev[q + 1][1], facs[q], None
                for _ in range(cycles):
                    v = mg(q + 1, v, res.reshape(4, Z, fac, X, fac).mean(dim=(2, 4)))
                v = v.repeat_interleave(fac, 1).repeat_interleave(fac, 2)
                x = -v if x is None else x - v
            x = smooth(x, rhs, dts[q], J, d if q == 0 else f)
            return torch.zeros_like(rhs) if x is None else x
        J = lambda y: jac(self.rhs, U, y)  # noqa: E731
        z = smooth(None, r, dtd, J, a)
        x = self.to_dg(mg(0, None, self.to_fv(r if z is None else r - J(z))))
        return smooth(x if z is None else z + x, r, dtd, J, b)


def exact(case, seed):
    if case["kind"] not in ("residual", "jv", "precond"):
        return None   # a step's result is defined up to the Newton tolerance only
    s = prepare(case, seed)
    pl, U = _Plain(case), s["U0"]
    shape = (4, pl.nz, pl.nx, pl.n1, pl.n1)
    if case["kind"] == "residual":
        return pl.rhs(U.reshape(shape)).reshape(-1)
    adt = ADT * _dt(case)
    if case["kind"] == "jv":
        y = s["y"]
        f1, f0 = (pl.rhs(A.reshape(shape)).reshape(-1) for A in (U + case["eps"] * y, U))
        return y - adt * (f1 - f0) / case["eps"]
    pre = getattr(presets, case["preset"]) if "preset" in case else {}
    return pl.precondition(U, adt, s["y"], pre.get("mg_key", case.get("key")), case["levels"], pre.get("sigma_fv", 1.0),
                           pre.get("sigma_dg", 1.0)).reshape(-1)
