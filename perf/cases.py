"""The workloads this library is timed on: what its users have it do, from the
smallest launch-bound run to the largest grid, through the public classes
(``Solver``, ``Batch``, ``LevelSet``) and the level-set entry points.

A case is a dict of plain values.  Its ``family`` says which entry point it
goes through:

- ``flow``: one grid.  ``op`` = "step" (set the state, advance ``steps``
  TVD-RK3 steps, read the state back), "rhs" (one right-hand side), "rhs_vjp"
  or "step_vjp" (reverse mode).
- ``batch``: ``nsim`` independent water drops of uneven sizes, ``steps`` steps
  of all of them.
- ``ls_step``: time steps of the two-phase level-set model.
- ``ls_transport``: level-set advection, reinitialisation and geometry.

``exact`` restates the method in plain float64 torch (no code of this
package): WENO5-JS / WENO5-Z / TENO6-A reconstruction, HLLC, central viscous
fluxes, limiters, THINC, TVD-RK3, and the level-set model.  Reverse mode is
torch autograd through that restatement.
"""
import math

import numpy as np
import torch

import paper_2402_05193_gb300 as jxf

DT = torch.float64
SIZES_BATCH = (64, 128, 192, 256)


# ----------------------------------------------------------------- cases ----
def _flow(name, **k):
    c = dict(family="flow", name=name, op="step", steps=1, model="spm", recon="char", weno="js", precision="fp64",
             viscous=False, visc_order=4, mu=0.0, limiter=False, thinc=False, nz=1, ny=1, ndim=3, gamma1=1.4,
             gamma2=1.4, pinf1=0.0, pinf2=0.0, cfl=0.5, bcx="periodic", bcy="periodic", bcz="periodic")
    c.update(k)
    return c


def listed():
    z = dict(bcx="zerograd", bcy="zerograd", bcz="zerograd")
    return [
        # a 1-D shock tube: every launch is small, latency and launch count decide
        _flow("tube_200_fp64", kind="tube", ndim=1, nx=200, recon="comp", steps=20, **z),
        # a small 2-D shear layer in float, many short steps (parameter studies, tests)
        _flow("shear_64x48_fp32", kind="shear", ndim=2, nx=64, ny=48, recon="comp", steps=10, precision="fp32"),
        # the library's headline run: viscous Taylor-Green vortex, both precisions
        _flow("vortex_128_fp64", kind="vortex", nx=128, ny=128, nz=128, viscous=True, mu=1.0 / 1600.0),
        _flow("vortex_128_fp32", kind="vortex", nx=128, ny=128, nz=128, viscous=True, mu=1.0 / 1600.0, steps=2,
              precision="fp32"),
        # TENO6-A with 6th-order viscous fluxes between walls, odd sizes: one right-hand side
        _flow("teno_walls_67x58x45_fp64", kind="smooth", op="rhs", nx=67, ny=58, nz=45, weno="teno6a", viscous=True,
              visc_order=6, mu=1e-2, bcx="symmetry", bcy="zerograd"),
        # air-helium shock-bubble interaction, five-equation model with limiters (mixed precision production run)
        _flow("bubble_256x128x128_fp32", kind="bubble", nx=256, ny=128, nz=128, model="dim", limiter=True, gamma2=1.66,
              cfl=0.4, precision="fp32", **z),
        # the same physics in double on a ragged 2-D grid, WENO5-Z and the THINC interface reconstruction
        _flow("bubble_thinc_301x150_fp64", kind="bubble", ndim=2, nx=301, ny=150, model="dim", limiter=True, thinc=True,
              weno="z", gamma2=1.66, cfl=0.4, steps=2, **z),
        # gradient of a rollout: the adjoint of one step on the Kelvin-Helmholtz grid
        _flow("shear_256_step_vjp_fp64", kind="shear", op="step_vjp", ndim=2, nx=256, ny=256),
        # an ensemble of shocked water drops of uneven sizes in one launch
        dict(family="batch", name="drops_24_fp32", nsim=24, steps=4, precision="fp32"),
        # the two-phase level-set model, one full time step (drop in a sound field)
        dict(family="ls_step", name="levelset_drop_96_fp64", ndim=3, nx=96, ny=96, nz=96, recon="js_char", steps=1,
             bc="periodic"),
        # level-set transport alone on a grid with odd sides
        dict(family="ls_transport", name="levelset_transport_125x110x131_fp64", ndim=3, nx=125, ny=110, nz=131,
             bc="zerograd"),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the listed ranges: any family, sizes spread over their
    logarithm, every option the listed cases use."""
    bcs = ("periodic", "zerograd", "symmetry")
    fam = rng.choice(("flow", "flow", "flow", "flow", "dim", "dim", "vjp", "batch", "ls_step", "ls_transport"))
    prec = rng.choice(("fp64", "fp32"))
    if fam == "flow":
        ndim = rng.choice((1, 2, 3, 3))
        total = _logint(rng, 200, 120 ** 3 if ndim == 3 else (500 * 500 if ndim == 2 else 20000))
        side = max(8, int(round(total ** (1.0 / ndim))))
        n = [max(7, int(side * rng.uniform(0.8, 1.25))) if e < ndim else 1 for e in range(3)]
        weno = rng.choice(("js", "js", "z", "teno6a"))
        viscous = rng.random() < 0.5
        op = rng.choice(("step", "rhs"))
        bc = [rng.choice(bcs) for _ in range(3)]
        return _flow("", kind="smooth", op=op, ndim=ndim, nx=n[0], ny=n[1], nz=n[2], weno=weno, viscous=viscous,
                     visc_order=rng.choice((2, 4, 6)), mu=10.0 ** rng.uniform(-4, -2) if viscous else 0.0,
                     recon=rng.choice(("comp", "char")), precision=prec, bcx=bc[0], bcy=bc[1], bcz=bc[2])
    if fam == "dim":
        ndim = rng.choice((1, 2, 3))
        total = _logint(rng, 200, 100 ** 3 if ndim == 3 else (400 * 400 if ndim == 2 else 4000))
        side = max(24, int(round(total ** (1.0 / ndim))))
        n = [max(20, int(side * rng.uniform(0.8, 1.25))) if e < ndim else 1 for e in range(3)]
        return _flow("", kind="bubble", model="dim", ndim=ndim, nx=n[0], ny=n[1], nz=n[2], limiter=True,
                     thinc=rng.random() < 0.4, weno=rng.choice(("js", "z")), gamma2=1.66, cfl=0.4, precision=prec,
                     op=rng.choice(("step", "rhs")), bcx="zerograd", bcy="zerograd", bcz="zerograd")
    if fam == "vjp":
        ndim = rng.choice((2, 3))
        total = _logint(rng, 500, 300 * 300)
        side = max(8, int(round(total ** (1.0 / ndim))))
        n = [max(7, int(side * rng.uniform(0.8, 1.25))) if e < ndim else 1 for e in range(3)]
        return _flow("", kind="shear" if ndim == 2 else "smooth", op=rng.choice(("rhs_vjp", "step_vjp")), ndim=ndim,
                     nx=n[0], ny=n[1], nz=n[2], weno=rng.choice(("js", "z")), recon=rng.choice(("comp", "char")),
                     precision=prec)
    if fam == "batch":
        return dict(family="batch", name="", nsim=_logint(rng, 2, 30), steps=rng.choice((1, 2, 3)), precision=prec)
    ndim = rng.choice((2, 3, 3))
    side = _logint(rng, 24, 96) if ndim == 3 else _logint(rng, 30, 400)
    n = [max(20, int(side * rng.uniform(0.85, 1.15))) if e < ndim else 1 for e in range(3)]
    if fam == "ls_step":
        return dict(family="ls_step", name="", ndim=ndim, nx=n[0], ny=n[1], nz=n[2], steps=1,
                    recon=rng.choice(("js_char", "z_char", "js_comp")), bc=rng.choice(("periodic", "zerograd")))
    return dict(family="ls_transport", name="", ndim=ndim, nx=n[0], ny=n[1], nz=n[2], bc=rng.choice(bcs))


# ---------------------------------------------------------------- inputs ----
def _n(case):
    return [case["nx"], case["ny"], case["nz"]][:case["ndim"]]


def _axes(case, length):
    n = _n(case)
    out = []
    for e in range(len(n)):
        x = (np.arange(n[e]) + 0.5) * (length[e] / n[e])
        shape = [1, 1, 1]
        shape[2 - e] = n[e]
        out.append(x.reshape(shape))
    return out


def _waves(rng, ax, length, amp, kmax=3):
    """Sum of three random plane-wave products with zero mean."""
    f = 0.0
    for _ in range(3):
        t = amp * rng.uniform(0.3, 1.0) / 3.0
        for x, ell in zip(ax, length):
            t = t * np.cos(2 * math.pi * rng.integers(0, kmax + 1) * x / ell + rng.uniform(0, 2 * math.pi))
        f = f + t
    return f


def _field(case, seed):
    """Primitive state (nv, nz, ny, nx) and the cell size per axis."""
    rng = np.random.default_rng(seed)
    n, nd = _n(case), case["ndim"]
    kind = case["kind"]
    one = np.ones((case["nz"], case["ny"], case["nx"]))
    if kind == "bubble":
        dx = 1e-3
        length = [m * dx for m in n]
        ax = _axes(case, length)
        s = n[0] / 256.0
        c = [(100.0 * s + rng.uniform(-2, 2)) * dx] + [(0.5 * n[e] + rng.uniform(-2, 2)) * dx for e in range(1, nd)]
        R = 25.0 * s * dx * rng.uniform(0.9, 1.1)
        r = np.sqrt(sum((ax[e] - c[e]) ** 2 for e in range(nd)))
        a = np.clip(0.5 * (1.0 + np.tanh((r - R) / dx)), 1e-8, 1.0 - 1e-8) * one
        post = ax[0] < 70.0 * s * dx + 0.0 * one
        w = 1.0 + _waves(rng, ax, length, 0.02)
        W = [a * np.where(post, 1.6573, 1.2041) * w, (1.0 - a) * 0.1660 * w]
        W += [np.where(post, 114.5, 0.0) * one if e == 0 else 5.0 * _waves(rng, ax, length, 1.0) * one
              for e in range(nd)]
        W += [np.where(post, 159056.0, 101325.0) * (1.0 + _waves(rng, ax, length, 0.02)), a]
        return np.stack([np.broadcast_to(w, one.shape) for w in W]), [dx] * nd
    if kind == "tube":
        length = [1.0]
        ax = _axes(case, length)
        left = ax[0] < rng.uniform(0.4, 0.6)
        W = [np.where(left, 1.0, 0.125) * (1.0 + _waves(rng, ax, length, 0.05)), 0.1 * _waves(rng, ax, length, 1.0),
             np.where(left, 1.0, 0.1) * (1.0 + _waves(rng, ax, length, 0.05))]
    elif kind == "shear":
        length = [1.0] * nd
        ax = _axes(case, length)
        br = np.tanh((ax[1] - 0.25) / 0.03) - np.tanh((ax[1] - 0.75) / 0.03)
        W = [1.0 + 0.5 * br + _waves(rng, ax, length, 0.05), -0.5 + 0.5 * br + _waves(rng, ax, length, 0.02),
             _waves(rng, ax, length, 0.05), 2.5 + _waves(rng, ax, length, 0.05)]
    elif kind == "vortex":
        length = [2.0 * math.pi] * nd
        X, Y, Z = _axes(case, length)
        p0 = 1.0 / (1.4 * 0.1 * 0.1)
        p = p0 + (np.cos(2 * X) + np.cos(2 * Y)) * (np.cos(2 * Z) + 2.0) / 16.0
        ax = [X, Y, Z]
        W = [p / p0 * (1.0 + _waves(rng, ax, length, 0.01)), np.sin(X) * np.cos(Y) * np.cos(Z),
             -np.cos(X) * np.sin(Y) * np.cos(Z), np.zeros_like(X), p]
        for e in range(3):
            W[1 + e] = W[1 + e] + _waves(rng, ax, length, 0.1)
    else:  # smooth
        length = [1.0] * nd
        ax = _axes(case, length)
        W = [1.0 + _waves(rng, ax, length, 0.2)] + [0.3 + _waves(rng, ax, length, 0.3) for _ in range(nd)] + \
            [1.0 + _waves(rng, ax, length, 0.2)]
    return np.stack([np.broadcast_to(w, one.shape) for w in W]), [length[e] / n[e] for e in range(nd)]


def _solver_case(case, dx, W=None):
    bc = [case["bcx"], case["bcy"], case["bcz"]]
    return dict(ndim=case["ndim"], n=_n(case), dx=dx, bc=[(b, b) for b in bc[:case["ndim"]]], model=case["model"],
                gamma=(case["gamma1"], case["gamma2"]), pinf=(case["pinf1"], case["pinf2"]), mu=case["mu"], Pr=0.72,
                R=1.0, recon=case["recon"], weno=case["weno"], viscous=case["viscous"],
                visc_order=case["visc_order"], limiter=case["limiter"], thinc=case["thinc"], cfl=case["cfl"],
                fixed_dt=0.0, t_end=0.0, W=W, f64=case["precision"] == "fp64")


def _drops(case, seed):
    """Shocked water drops in air, sizes from SIZES_BATCH."""
    rng = np.random.default_rng(seed)
    out = []
    for k in range(case["nsim"]):
        N = int(SIZES_BATCH[k % 4])
        dx = 1.0 / N
        x = (np.arange(N) + 0.5) * dx
        Y, X = np.meshgrid(x, x, indexing="ij")
        radius, cx, cy = rng.uniform(0.08, 0.15), rng.uniform(0.4, 0.6), rng.uniform(0.35, 0.65)
        m2 = rng.uniform(1.2, 2.4) ** 2
        a = np.clip(0.5 * (1.0 - np.tanh((np.hypot(X - cx, Y - cy) - radius) / dx)), 1e-8, 1.0 - 1e-8)
        rho2, p2 = 1.2 * 2.4 * m2 / (0.4 * m2 + 2.0), 1.01e5 * (1.0 + 2.8 / 2.4 * (m2 - 1.0))
        u2 = math.sqrt(m2 * 1.4 * 1.01e5 / 1.2) * (1.0 - 1.2 / rho2)
        post = X < cx - radius - 0.05
        ax = [x.reshape(1, 1, N), x.reshape(1, N, 1)]
        w, v = [_waves(rng, ax, [1.0, 1.0], s)[0] for s in (0.03, 30.0)]
        W = np.stack([a * 1000.0, (1.0 - a) * np.where(post, rho2, 1.2) * (1.0 + w),
                      np.where(post, u2, 0.0) * (1.0 + w), (1.0 - a) * v, np.where(post, p2, 1.01e5) * (1.0 + w),
                      a])[:, None]
        out.append(dict(ndim=2, n=[N, N], dx=[dx, dx], bc=[("zerograd", "zerograd")] * 2, model="dim",
                        gamma=(6.12, 1.4), pinf=(3.43e8, 0.0), mu=0.0, Pr=0.72, R=1.0, recon="char", weno="js",
                        viscous=False, visc_order=4, limiter=True, thinc=False, cfl=0.4, fixed_dt=0.0, t_end=0.0,
                        W=np.ascontiguousarray(W), f64=case["precision"] == "fp64"))
    return out


def _levelset(case, seed):
    """phi, W1, W2 of a drop (ellipsoid, signed distance distorted by a few per
    cent as between reinitialisations) in a sound field; cubic cells."""
    rng = np.random.default_rng(seed)
    n, nd = _n(case), case["ndim"]
    h = 1.0 / max(n)
    length = [m * h for m in n]
    ax = _axes(case, length)
    one = np.ones((case["nz"], case["ny"], case["nx"]))
    c = [ell * rng.uniform(0.45, 0.55) for ell in length]
    R = 0.25 * min(length)
    r = np.sqrt(sum((ax[e] - c[e]) ** 2 for e in range(nd)))
    phi = (R - r) * (1.0 + _waves(rng, ax, length, 0.03)) * one

    def prim(rho, p):
        w = [rho * (1.0 + _waves(rng, ax, length, 0.05))]
        w += [u + _waves(rng, ax, length, 0.1) for u in (0.4, 0.3, 0.2)[:nd]]
        return np.stack([a * one for a in w + [p * (1.0 + _waves(rng, ax, length, 0.05))]])

    W1, W2 = prim(5.0, 1.0), prim(1.0, 1.0)
    vel = np.stack([(u + _waves(rng, ax, length, 0.5)) * one for u in (0.4, -0.3, 0.2)[:nd]])
    sh = one.shape if nd == 3 else one.shape[1:]
    return (phi.reshape(sh), W1.reshape((nd + 2,) + sh), W2.reshape((nd + 2,) + sh), vel.reshape((nd,) + sh), h,
            0.3 * h / (0.75 + math.sqrt(4.4 * 7.0 / 5.0)))


_LS_MAT = ((4.4, 6.0), (1.4, 0.0))
_BC = {"periodic": 0, "zerograd": 1, "symmetry": 2}


def _ls_bc(case):
    b = _BC[case["bc"]]
    return [(b, b)] * case["ndim"]


def _adjoint_seed(case, seed, U):
    rng = np.random.default_rng(seed + 7919)
    g = torch.from_numpy(rng.standard_normal(tuple(U.shape))).to(U.device)
    return g.to(U.dtype)


def prepare(case, seed):
    dev = "cuda"
    fam = case["family"]
    if fam == "flow":
        W, dx = _field(case, seed)
        sc = _solver_case(case, dx)
        U = _cons(sc, torch.from_numpy(np.ascontiguousarray(W)))
        U = U.to(DT if sc["f64"] else torch.float32).to(dev).contiguous()
        st = dict(case=case, solver=jxf.Solver(sc, case["precision"]), U=U, dt=_vjp_dt(case, dx))
        if case["op"].endswith("vjp"):
            st["bar"] = _adjoint_seed(case, seed, U)
        return st
    if fam == "batch":
        cs = _drops(case, seed)
        b = jxf.Batch(cs, case["precision"])
        dt = DT if case["precision"] == "fp64" else torch.float32
        U = [_cons(c, torch.from_numpy(c["W"])).to(dt).to(dev).contiguous() for c in cs]
        return dict(case=case, batch=b, U=U)
    phi, W1, W2, vel, h, dt = _levelset(case, seed)
    t = [torch.from_numpy(np.ascontiguousarray(a)).to(dev) for a in (phi, W1, W2, vel)]
    if fam == "ls_step":
        ls = jxf.LevelSet(case["ndim"], _n(case), h, _ls_bc(case), _LS_MAT[0], _LS_MAT[1], case["recon"])
        return dict(case=case, ls=ls, fields=t[:3], dt=dt)
    grid = jxf.ls_grid(case["ndim"], _n(case), h, _ls_bc(case))
    nc = t[0].numel()
    z = lambda *s: torch.zeros(s, dtype=DT, device=dev)  # noqa: E731
    return dict(case=case, grid=grid, phi0=t[0], vel=t[3], phi=z(*t[0].shape), scratch=z(2 * nc),
                ap=z(jxf.jxf_ls_nface(grid)), al=z(*t[0].shape), dg=z(*t[0].shape),
                nr=z(case["ndim"], *t[0].shape), dt=0.3 * h)


def _vjp_dt(case, dx):
    return 0.1 * min(dx)


def run(state):
    case = state["case"]
    fam = case["family"]
    if fam == "flow":
        s, U, op = state["solver"], state["U"], case["op"]
        if op == "step":
            s.set_state(U)
            s.step(case["steps"], sync=False)
            return s.state()
        if op == "rhs":
            return s.rhs(U, state["dt"])
        if op == "rhs_vjp":
            return s.rhs_vjp(U, state["bar"])
        return s.step_vjp(U, state["dt"], state["bar"])
    if fam == "batch":
        b = state["batch"]
        for k, U in enumerate(state["U"]):
            jxf.jxf_batch_set_state(b.b, k, U)
        b.step(case["steps"])
        return [b.state(k) for k in range(case["nsim"])]
    if fam == "ls_step":
        ls = state["ls"]
        ls.set_state(*state["fields"])
        ls.step(state["dt"], case["steps"])
        return [ls.phi, ls.aU1, ls.aU2, ls.W1, ls.W2, ls.qg]
    g, phi = state["grid"], state["phi"]
    phi.copy_(state["phi0"])
    jxf.jxf_ls_advect(g, phi, state["vel"], state["dt"], 1, state["scratch"])
    jxf.jxf_ls_reinit(g, phi, 10, 5e-2, state["scratch"])
    jxf.jxf_ls_geometry(g, phi, state["ap"], state["al"], state["dg"], state["nr"])
    return [phi, state["ap"], state["al"], state["dg"], state["nr"]]


# Operations per cell of one face sweep (one axis), counted on the scheme's
# plain formulas: WENO5 per variable and face, projection and HLLC, TENO6-A's
# larger stencil work, the viscous flux.
def _sweep_flops(case):
    nv = case["ndim"] + (4 if case["model"] == "dim" else 2)
    per = 500 if case["weno"] == "teno6a" else 120
    f = per * nv + 160 + (60 * nv if case["recon"] == "char" else 0) + (150 if case["viscous"] else 0)
    return f + (200 if case["limiter"] else 0)


def work(case):
    fam = case["family"]
    if fam == "batch":
        cells = sum(SIZES_BATCH[k % 4] ** 2 for k in range(case["nsim"]))
        es = 8 if case["precision"] == "fp64" else 4
        return {"bytes": 2 * 6 * es * cells, "flops": 7956.0 * cells * case["steps"]}
    cells = 1
    for m in _n(case):
        cells *= m
    nd = case["ndim"]
    if fam == "flow":
        es = 8 if case["precision"] == "fp64" else 4
        nv = nd + (4 if case["model"] == "dim" else 2)
        per_rhs = nd * _sweep_flops(case) + 20 * nv
        k = {"step": 3 * case["steps"], "rhs": 1, "rhs_vjp": 3, "step_vjp": 11}[case["op"]]
        arrays = 3 if case["op"].endswith("vjp") else 2
        return {"bytes": arrays * nv * es * cells, "flops": float(per_rhs * k * cells)}
    if fam == "ls_transport":
        return {"bytes": 8 * cells * (2 + nd + nd + 2 + nd), "flops": 4200.0 * cells * nd / 3}
    nv = nd + 2
    # one phase's face fluxes per cell, 20 reinitialisation stages, the extensions
    per = 3 * (nd * 900 + 10 * nv * 8 + 20 * (nd + 1) * 8 + 170) + 20 * 65 * nd
    return {"bytes": 8 * cells * (2 * (1 + 2 * nv) + 2 * nv + nd + 1), "flops": float(per * cells * case["steps"])}


# ------------------------------------------------- the method in float64 ----
# Arrays (variable, z, y, x); axis e is tensor dimension -1 - e.
def _np_of(c):
    return 2 if c["model"] == "dim" else 1


def _ab(c, a1):
    """A = 1/(gamma-1), B = gamma p_inf/(gamma-1) of the mixture."""
    g, p = c["gamma"], c["pinf"]
    A = [1.0 / (x - 1.0) for x in g]
    B = [x * y / (x - 1.0) for x, y in zip(g, p)]
    if c["model"] != "dim":
        return A[0], B[0]
    return a1 * A[0] + (1.0 - a1) * A[1], a1 * B[0] + (1.0 - a1) * B[1]


def _rho(c, X):
    return X[0] + X[1] if c["model"] == "dim" else X[0]


def _rc2(c, W):
    nd, q = c["ndim"], _np_of(c)
    p = W[q + nd]
    if c["model"] != "dim":
        return c["gamma"][0] * (p + c["pinf"][0])
    A, B = _ab(c, W[q + nd + 1])
    return p + (p + B) / A


def _cons(c, W):
    nd, q = c["ndim"], _np_of(c)
    rho = _rho(c, W)
    A, B = _ab(c, W[q + nd + 1] if c["model"] == "dim" else None)
    U = [W[k] for k in range(q)] + [rho * W[q + e] for e in range(nd)]
    uu = sum(W[q + e] * W[q + e] for e in range(nd))
    U.append(A * W[q + nd] + B + 0.5 * rho * uu)
    if c["model"] == "dim":
        U.append(W[q + nd + 1])
    return torch.stack(U)


def _prim(c, U):
    nd, q = c["ndim"], _np_of(c)
    rho = _rho(c, U)
    u = [U[q + e] / rho for e in range(nd)]
    A, B = _ab(c, U[q + nd + 1] if c["model"] == "dim" else None)
    p = (U[q + nd] - 0.5 * rho * sum(x * x for x in u) - B) / A
    W = [U[k] for k in range(q)] + u + [p]
    if c["model"] == "dim":
        W.append(U[q + nd + 1])
    return torch.stack(W)


def _mapped(n, g, bc, device):
    """Indices of cells -g .. n+g-1 through the boundary conditions, and which
    of them are mirrored."""
    k = torch.arange(-g, n + g, device=device)
    if bc == "periodic":
        return k % n, torch.zeros_like(k, dtype=torch.bool)
    if bc == "zerograd":
        return k.clamp(0, n - 1), torch.zeros_like(k, dtype=torch.bool)
    m = (k < 0) | (k >= n)
    return torch.where(k < 0, -1 - k, torch.where(k >= n, 2 * n - 1 - k, k)), m


def _ghost(a, e, g, bc, flip=None):
    """a with g mapped cells on both sides of axis e; rows `flip` of the first
    dimension change sign in mirrored cells."""
    dim = a.dim() - 1 - e
    idx, mir = _mapped(a.shape[dim], g, bc, a.device)
    out = a.index_select(dim, idx)
    if flip and bc == "symmetry":
        s = torch.where(mir, -1.0, 1.0).to(a.dtype).reshape([-1] + [1] * e)
        out = torch.stack([out[v] * s if v in flip else out[v] for v in range(out.shape[0])])
    return out


def _win(a, e, j, m):
    return a.narrow(a.dim() - 1 - e, j, m)


def _weno5_left(v, z, eps=1e-6):
    a, b, c, d, e = v
    q = ((2 * a - 7 * b + 11 * c) / 6, (-b + 5 * c + 2 * d) / 6, (2 * c + 5 * d - e) / 6)
    k = 13.0 / 12.0
    s = (k * (a - 2 * b + c) ** 2 + 0.25 * (a - 4 * b + 3 * c) ** 2, k * (b - 2 * c + d) ** 2 + 0.25 * (b - d) ** 2,
         k * (c - 2 * d + e) ** 2 + 0.25 * (3 * c - 4 * d + e) ** 2)
    if z:
        tau = (s[0] - s[2]).abs()
        w = [dk * (1.0 + tau / (sk + eps)) for dk, sk in zip((0.1, 0.6, 0.3), s)]
    else:
        w = [dk / (sk + eps) ** 2 for dk, sk in zip((0.1, 0.6, 0.3), s)]
    return (w[0] * q[0] + w[1] * q[1] + w[2] * q[2]) / (w[0] + w[1] + w[2])


def _teno_left(v):
    a, b, c, d, e, f = v
    q = ((-b + 5 * c + 2 * d) / 6, (2 * c + 5 * d - e) / 6, (2 * a - 7 * b + 11 * c) / 6,
         (3 * c + 13 * d - 5 * e + f) / 12)
    k = 13.0 / 12.0
    e1, e2 = -11 * c + 18 * d - 9 * e + 2 * f, 2 * c - 5 * d + 4 * e - f
    e3 = -c + 3 * d - 3 * e + f
    s = (k * (b - 2 * c + d) ** 2 + 0.25 * (b - d) ** 2, k * (c - 2 * d + e) ** 2 + 0.25 * (3 * c - 4 * d + e) ** 2,
         k * (a - 2 * b + c) ** 2 + 0.25 * (a - 4 * b + 3 * c) ** 2,
         e1 * e1 / 36 + k * e2 * e2 + 781.0 / 720.0 * e3 * e3)
    # smoothness of the six-cell polynomial from its derivative coefficients
    a1 = (341 * a - 2785 * b - 2590 * c + 6670 * d - 1895 * e + 259 * f) / 5760
    a2 = (-a + 12 * b - 22 * c + 12 * d - e) / 16
    a3 = (-5 * a - 11 * b + 70 * c - 94 * d + 47 * e - 7 * f) / 144
    a4 = (a - 4 * b + 6 * c - 4 * d + e) / 24
    a5 = (-a + 5 * b - 10 * c + 10 * d - 5 * e + f) / 120
    t1, t2, t3 = a1 + a3 / 4 + a5 / 16, a2 + 63.0 / 130.0 * a4, a3 + 8825.0 / 10934.0 * a5
    s6 = t1 * t1 + 13.0 / 3.0 * t2 * t2 + 781.0 / 20.0 * t3 * t3 + 1421461.0 / 2275.0 * a4 * a4 + \
        21520059541.0 / 1377684.0 * a5 * a5
    tau = (s6 - (s[0] + s[2] + 4 * s[1]) / 6).abs()
    g = [(1.0 + tau / (x + 1e-30)) ** 6 for x in s]
    tot = g[0] + g[1] + g[2] + g[3]
    Cr, xi = 0.23, 1e-3
    e0 = 0.9 * Cr * xi * xi / (1.0 - 0.9 * Cr)
    eta = torch.ones_like(a)
    for j in range(1, 5):
        dp, dm = v[j + 1] - v[j], v[j] - v[j - 1]
        eta = torch.minimum(eta, ((2 * dp * dm).abs() + e0) / (dp * dp + dm * dm + e0))
    m = 1.0 - (eta / Cr).clamp(max=1.0)
    ct = 10.0 ** (-torch.floor(10.5 - 3.5 * (1.0 - (1.0 - m) ** 4 * (1.0 + 4.0 * m))))
    num, den = 0.0, 0.0
    for dk, gk, qk in zip((0.45, 0.3, 0.05, 0.2), g, q):
        keep = torch.where(gk / tot < ct, 0.0 * gk, torch.full_like(gk, dk))
        num, den = num + keep * qk, den + keep
    return num / den


def _sides(c, v):
    """Left and right face values from the six cells v."""
    if c["weno"] == "teno6a":
        return _teno_left(v), _teno_left(v[::-1])
    z = c["weno"] == "z"
    return _weno5_left(v[:5], z), _weno5_left(v[:0:-1], z)


def _reconstruct(c, S, d):
    """Face states from the stencil S (six states, lists of variables)."""
    nd, q = c["ndim"], _np_of(c)
    nv, ie, iu = len(S[0]), q + nd, q + d
    if c["recon"] != "char":
        out = [_sides(c, [S[j][v] for j in range(6)]) for v in range(nv)]
        return [o[0] for o in out], [o[1] for o in out]
    M = [0.5 * (x + y) for x, y in zip(S[2], S[3])]
    rho, rc2 = _rho(c, M), _rc2(c, M)
    cb = torch.sqrt(rc2 / rho)
    L, R = [None] * nv, [None] * nv
    for v in range(nv):
        if v < q:
            x = [S[j][v] - M[v] * S[j][ie] / rc2 for j in range(6)]
        elif v == ie or v == iu:
            sg = 1.0 if v == ie else -1.0
            x = [sg * S[j][iu] / (2.0 * cb) + S[j][ie] / (2.0 * rc2) for j in range(6)]
        else:
            x = [S[j][v] for j in range(6)]
        L[v], R[v] = _sides(c, x)
    for X in (L, R):
        m, p = X[iu], X[ie]
        for k in range(q):
            X[k] = X[k] + M[k] * (m + p)
        X[iu], X[ie] = cb * (p - m), rc2 * (m + p)
    return L, R


def _hllc(c, L, R, d):
    nd, q = c["ndim"], _np_of(c)
    ie, iu = q + nd, q + d
    rl, rr, ul, ur, pl, pr = _rho(c, L), _rho(c, R), L[iu], R[iu], L[ie], R[ie]
    c2l, c2r = _rc2(c, L) / rl, _rc2(c, R) / rr
    cl, cr = torch.sqrt(c2l), torch.sqrt(c2r)
    sl, sr = torch.sqrt(rl), torch.sqrt(rr)
    ub = (sl * ul + sr * ur) / (sl + sr)
    cb = torch.sqrt((sl * c2l + sr * c2r) / (sl + sr) + 0.5 * sl * sr / (sl + sr) ** 2 * (ur - ul) ** 2)
    SL = torch.where(ul - cl < ub - cb, ul - cl, ub - cb)
    SR = torch.where(ur + cr > ub + cb, ur + cr, ub + cb)
    ml, mr = rl * (SL - ul), rr * (SR - ur)
    ss = (pr - pl + ml * ul - mr * ur) / (ml - mr)
    sm, sp = torch.where(SL < 0.0, SL, 0.0 * SL), torch.where(SR > 0.0, SR, 0.0 * SR)

    def branch(X, s, spm):
        U = _cons(c, torch.stack(X) if isinstance(X, list) else X)
        rho, u, p = _rho(c, X), X[iu], X[ie]
        f = (s - u) / (s - ss)
        star = [f * x for x in U]
        star[iu] = f * rho * ss
        star[ie] = f * (U[ie] + (ss - u) * (rho * ss + p / (s - u)))
        F = [x * u for x in U]
        F[iu] = F[iu] + p
        F[ie] = u * (U[ie] + p)
        return [F[v] + spm * (star[v] - U[v]) for v in range(len(F))], u + spm * (f - 1.0)

    FL, hl = branch(L, SL, sm)
    FR, hr = branch(R, SR, sp)
    pick = lambda a, b: torch.where(ss > 0.0, a, torch.where(ss < 0.0, b, 0.5 * (a + b)))  # noqa: E731
    return torch.stack([pick(a, b) for a, b in zip(FL, FR)]), pick(hl, hr)


def _thinc_normal(c, W, dx):
    a = W[-1].clamp(0.0, 1.0)
    r = ((1.0 - a) / a) ** 0.1
    psi = torch.where(a > 0.0, 1.0 / (1.0 + r), 0.0 * a)[None]
    g = []
    for e in range(c["ndim"]):
        p = _ghost(psi, e, 1, c["bc"][e][0])
        m = W.shape[-1 - e]
        g.append((_win(p, e, 2, m) - _win(p, e, 0, m))[0] * (0.5 / dx[e]))
    nrm = torch.sqrt(sum(x * x for x in g))
    return torch.stack([torch.where(nrm > 0.0, x.abs() / nrm.clamp(min=1e-300), 0.0 * x) for x in g])


def _thinc_side(am, ac, ap, nabs, side, Wc, Wf):
    on = (ac >= 1e-4) & (ac <= 1.0 - 1e-4) & ((ap - ac) * (ac - am) > 0.0)
    up = ap > am
    beta = nabs + 0.01
    s = torch.where(up, 2.0 * ac - 1.0, 1.0 - 2.0 * ac)
    u, w = beta * (1.0 + s), beta * (1.0 - s)
    e = torch.exp(w) * torch.expm1(u) / torch.expm1(w) if side == 0 else \
        torch.expm1(u) / (torch.exp(u) * torch.expm1(w))
    a = torch.where(up, e / (e + 1.0), 1.0 / (e + 1.0))
    Wf = list(Wf)
    Wf[0] = torch.where(on, a * Wc[0] / ac, Wf[0])
    Wf[1] = torch.where(on, (1.0 - a) * Wc[1] / (1.0 - ac), Wf[1])
    Wf[-1] = torch.where(on, a, Wf[-1])
    return Wf


def _bad(c, X, rc2, eps):
    bad = rc2 < eps[1]
    for k in range(_np_of(c)):
        bad = bad | (X[k] < eps[0])
    if c["model"] == "dim":
        bad = bad | (X[-1] < eps[2]) | (X[-1] > 1.0 - eps[2])
    return bad


def _stencil_dn(v, h):
    if h == 1:
        return v[1] - v[0]
    if h == 2:
        return (v[0] - v[3] + 27 * (v[2] - v[1])) / 24
    return (9 * (v[5] - v[0]) + 125 * (v[1] - v[4]) + 2250 * (v[3] - v[2])) / 1920


def _stencil_val(v, h):
    if h == 1:
        return 0.5 * (v[0] + v[1])
    if h == 2:
        return (9 * (v[1] + v[2]) - (v[0] + v[3])) / 16
    return (150 * (v[2] + v[3]) - 25 * (v[1] + v[4]) + 3 * (v[0] + v[5])) / 256


def _cell_grad(c, W, dx, h):
    """du_f/dx_e at the cell centres."""
    nd = c["ndim"]
    G = {}
    for e in range(nd):
        p = _ghost(W[1:1 + nd], e, h, c["bc"][e][0], [e])
        m = W.shape[-1 - e]
        w = [_win(p, e, k, m) for k in range(2 * h + 1)]
        if h == 1:
            g = (w[2] - w[0]) / 2
        elif h == 2:
            g = (w[0] - w[4] + 8 * (w[3] - w[1])) / 12
        else:
            g = (w[6] - w[0] + 9 * (w[1] - w[5]) + 45 * (w[4] - w[2])) / 60
        for f in range(nd):
            G[f, e] = g[f] / dx[e]
    return G


def _viscous(c, W, dx, d, S):
    nd, h = c["ndim"], c["visc_order"] // 2
    bc, m = c["bc"][d][0], W.shape[-1 - d] + 1
    j0 = 3 - h
    G = _cell_grad(c, W, dx, h)

    def faces(a, flip):
        p = _ghost(a[None], d, 3, bc, [0] if flip else None)[0]
        return [_win(p, d, j0 + k, m) for k in range(2 * h)]

    T = W[1 + nd] / (W[0] * c["R"])
    dn = [_stencil_dn([S[j0 + k][1 + f] for k in range(2 * h)], h) / dx[d] for f in range(nd)]
    u = [_stencil_val([S[j0 + k][1 + f] for k in range(2 * h)], h) for f in range(nd)]
    div = dn[d] + sum(_stencil_val(faces(G[e, e], False), h) for e in range(nd) if e != d)
    F = [0.0 * div]
    lam = c["mu"] * c["gamma"][0] * c["R"] / (c["gamma"][0] - 1.0) / c["Pr"]
    en = lam * _stencil_dn(faces(T, False), h) / dx[d]
    for k in range(nd):
        if k == d:
            tau = c["mu"] * (2.0 * dn[d] - 2.0 / 3.0 * div)
        else:
            tau = c["mu"] * (_stencil_val(faces(G[d, k], True), h) + dn[k])
        F.append(tau)
        en = en + u[k] * tau
    return torch.stack(F + [en])


def _flux(c, W, U, dx, d, dt, G=None):
    nd, q = c["ndim"], _np_of(c)
    bc, m = c["bc"][d][0], W.shape[-1 - d] + 1
    p = _ghost(W, d, 3, bc, [q + d])
    S = [list(_win(p, d, j, m)) for j in range(6)]
    L, R = _reconstruct(c, S, d)
    if c["thinc"]:
        gn = _ghost(G[d][None], d, 3, bc)[0]
        L = _thinc_side(S[1][-1], S[2][-1], S[3][-1], _win(gn, d, 2, m), 0, S[2], L)
        R = _thinc_side(S[2][-1], S[3][-1], S[4][-1], _win(gn, d, 3, m), 1, S[3], R)
    if c["limiter"]:
        eps = (1e-12, 1e-10, 1e-12) if c["f64"] else (1e-10, 1e-8, 1e-10)
        out = []
        for X, C in ((L, S[2]), (R, S[3])):
            bad = _bad(c, X, _rc2(c, X), eps)
            out.append([torch.where(bad, y, x) for x, y in zip(X, C)])
        L, R = out
    F, uh = _hllc(c, L, R, d)
    if c["limiter"]:
        pu = _ghost(U, d, 1, bc, [q + d])
        lam = 2.0 * nd / dx[d] * dt
        bad = torch.zeros_like(F[0], dtype=torch.bool)
        for s, j in ((-1.0, 0), (1.0, 1)):
            Uc = _win(pu, d, j, m)
            T = Uc + s * lam * F
            T = torch.cat([T[:-1], (Uc[-1] + s * lam * (F[-1] - Uc[-1] * uh))[None]])
            bad = bad | _bad(c, T, _rc2(c, _prim(c, T)), eps)
        F1, uh1 = _hllc(c, S[2], S[3], d)
        F, uh = torch.where(bad, F1, F), torch.where(bad, uh1, uh)
    if c["viscous"]:
        F = F - _viscous(c, W, dx, d, S)
    return F, uh


def _rhs(c, U, dt):
    dx = c["dx"]
    W = _prim(c, U)
    G = _thinc_normal(c, W, dx) if c["thinc"] else None
    R = torch.zeros_like(U)
    for d in range(c["ndim"]):
        F, uh = _flux(c, W, U, dx, d, dt, G)
        m = U.shape[-1 - d]
        R = R - (_win(F, d, 1, m) - _win(F, d, 0, m)) / dx[d]
        if c["model"] == "dim":
            src = U[-1] * (_win(uh, d, 1, m) - _win(uh, d, 0, m)) / dx[d]
            R = torch.cat([R[:-1], (R[-1] + src)[None]])
    return R


def _cfl(c, U):
    W = _prim(c, U)
    q = _np_of(c)
    rho = _rho(c, W)
    cs = torch.sqrt(_rc2(c, W) / rho)
    dt = c["cfl"] / float(sum((W[q + e].abs() + cs) / c["dx"][e] for e in range(c["ndim"])).max())
    if c["viscous"] and c["mu"] > 0.0:
        dt = min(dt, c["cfl"] * 3.0 / 14.0 * float(rho.min()) * min(c["dx"]) ** 2 / c["mu"])
    return dt


def _rk3(c, U, dt):
    U1 = U + dt * _rhs(c, U, dt)
    U2 = 0.75 * U + 0.25 * U1 + 0.25 * dt * _rhs(c, U1, dt)
    return U / 3.0 + 2.0 / 3.0 * U2 + 2.0 / 3.0 * dt * _rhs(c, U2, dt)


def _advance(c, U, steps):
    for _ in range(steps):
        U = _rk3(c, U, _cfl(c, U))
    return U


# -------------------------------------------- the level-set model in float64 --
def _sh(a, e, s, bc):
    """a at the cell moved by s along axis e."""
    g = abs(s)
    return _win(_ghost(a, e, g, bc), e, g + s, a.shape[a.dim() - 1 - e]) if s else a


def _ls_fraction(p):
    pos = [x > 0.0 for x in p]
    n = sum(x.to(torch.int8) for x in pos)
    safe = lambda a, b: a / torch.where(a == b, torch.ones_like(a), a - b)  # noqa: E731
    tn = [safe(p[k], p[(k + 1) & 3]) for k in range(4)]
    tp = [safe(p[k], p[(k + 3) & 3]) for k in range(4)]
    out = torch.where(n == 4, 1.0, 0.0).to(DT)
    tri = [0.5 * tn[k] * tp[k] for k in range(4)]
    for k in range(4):
        a, b = (k + 1) & 3, (k + 2) & 3
        out = torch.where((n == 1) & pos[k], tri[k], out)
        out = torch.where((n == 3) & ~pos[k], 1.0 - tri[k], out)
        out = torch.where((n == 2) & pos[k] & pos[a], 0.5 * (tp[k] + tn[a]), out)
        out = torch.where((n == 2) & pos[k] & pos[b], tri[k] + tri[b], out)
    return out


def _ls_geometry(phi, h, bc):
    nd = phi.dim()
    P = phi
    for e in range(nd):
        P = _ghost(P, e, 1, bc)
    n = [phi.shape[-1 - e] for e in range(nd)]
    V = torch.zeros_like(P[tuple(slice(0, m + 1) for m in reversed(n))])
    for k in range(2 ** nd):  # x fastest, the summation order of the vertex mean
        V = V + P[tuple(slice((k >> e) & 1, ((k >> e) & 1) + n[e] + 1) for e in reversed(range(nd)))]
    V = V / float(2 ** nd)
    A, lo, hi = [], [], []
    for d in range(nd):
        t = [e for e in range(nd) if e != d]
        corner = (((0, 0), (1, 0), (1, 1), (0, 1)) if nd == 3 else ((0,), (1,)))
        p = []
        for off in corner:
            v = V
            for e, o in zip(t, off):
                v = _win(v, e, o, n[e])
            p.append(v)
        if nd == 3:
            f = _ls_fraction(p)
        else:
            a, b = p
            pa, pb = a > 0.0, b > 0.0
            dif = torch.where(a == b, torch.ones_like(a), a - b)
            f = torch.where(pa & pb, 1.0, torch.where(pa, a / dif, torch.where(pb, -b / dif, 0.0 * a)))
        A.append(f)
        lo.append(_win(f, d, 0, n[d]))
        hi.append(_win(f, d, 1, n[d]))
    S, vol = h ** (nd - 1), h ** nd
    dg = torch.sqrt(sum(((b - a) * S) ** 2 for a, b in zip(lo, hi)))
    al = ((sum((a + b) * S * 0.5 * h for a, b in zip(lo, hi)) + dg * phi) / (nd * vol)).clamp(0.0, 1.0)
    g = [(_sh(phi, e, -2, bc) - 8 * _sh(phi, e, -1, bc) + 8 * _sh(phi, e, 1, bc) - _sh(phi, e, 2, bc)) / (12 * h)
         for e in range(nd)]
    m = torch.sqrt(sum(x * x for x in g))
    nr = torch.stack([torch.where(m > 0.0, x / m.clamp(min=1e-300), 0.0 * x) for x in g])
    return A, al, dg, nr


def _ls_advect_rhs(phi, vel, h, bc):
    r = torch.zeros_like(phi)
    for d in range(phi.dim()):
        s = {k: _sh(phi, d, k, bc) for k in range(-3, 4)}
        left = (-2 * s[-3] + 15 * s[-2] - 60 * s[-1] + 20 * s[0] + 30 * s[1] - 3 * s[2]) / (60 * h)
        right = (3 * s[-2] - 30 * s[-1] - 20 * s[0] + 60 * s[1] - 15 * s[2] + 2 * s[3]) / (60 * h)
        r = r - vel[d] * torch.where(vel[d] >= 0.0, left, right)
    return r


def _ls_reinit_rhs(phi, phi0, h, bc, thr):
    sg = torch.sign(phi0)
    pos = phi0 > 0.0

    def weno3(a, b, c):
        s0, s1 = 1e-6 + (b - a) ** 2, 1e-6 + (c - b) ** 2
        w0, w1 = 1.0 / (3.0 * s0 * s0), 2.0 / (3.0 * s1 * s1)
        return (w0 * (3 * b - a) / 2 + w1 * (b + c) / 2) / (w0 + w1)

    H = torch.zeros_like(phi)
    for d in range(phi.dim()):
        s = {k: _sh(phi, d, k, bc) for k in range(-2, 3)}
        D = [(s[k + 1] - s[k]) / h for k in range(-2, 2)]
        a, b = weno3(D[0], D[1], D[2]), weno3(D[3], D[2], D[1])
        t1 = torch.where(pos, a.clamp(min=0.0), a.clamp(max=0.0))
        t2 = torch.where(pos, b.clamp(max=0.0), b.clamp(min=0.0))
        H = H + torch.maximum(t1 * t1, t2 * t2)
    R = -sg * (torch.sqrt(H) - 1.0)
    return torch.where(R.abs() > thr, R, 0.0 * R)


def _ls_reinit(phi, h, bc, steps, thr=5e-2):
    phi0, dtau = phi, 0.25 * h
    for _ in range(steps):
        p1 = phi + dtau * _ls_reinit_rhs(phi, phi0, h, bc, thr)
        phi = 0.5 * phi + 0.5 * (p1 + dtau * _ls_reinit_rhs(p1, phi0, h, bc, thr))
    return phi


def _ls_extend(q, phi, al, dg, nr, mode, steps, bc):
    if mode == 0:
        sdir, fixed = -torch.ones_like(phi), al > 0.0
    elif mode == 1:
        sdir, fixed = torch.ones_like(phi), al < 1.0
    else:
        sdir, fixed = torch.sign(phi), ((al > 0.0) & (al < 1.0)) | (dg > 0.0)
    a = sdir * nr
    for _ in range(steps):
        r = q
        for d in range(phi.dim()):
            w = 0.25 * a[d].abs()
            up = torch.where(a[d] > 0.0, _sh(q, d, -1, bc), torch.where(a[d] < 0.0, _sh(q, d, 1, bc), q))
            r = r + w * (up - q)
        q = torch.where(fixed, q, r)
    return q


def _ls_interface(W1, W2, al, dg, nr):
    nd = nr.shape[0]
    cut = ((al > 0.0) & (al < 1.0)) | (dg > 0.0)
    Z, un, p = [], [], []
    for W, (g, pi) in zip((W1, W2), _LS_MAT):
        Z.append(W[0] * torch.sqrt(g * (W[1 + nd] + pi) / W[0]))
        un.append(sum(W[1 + e] * nr[e] for e in range(nd)))
        p.append(W[1 + nd])
    zs = Z[0] + Z[1]
    u = (Z[0] * un[0] + Z[1] * un[1] + p[1] - p[0]) / zs
    pg = (Z[0] * p[1] + Z[1] * p[0] + Z[0] * Z[1] * (un[1] - un[0])) / zs
    q = torch.cat([u * nr, pg[None]])
    return torch.where(cut, q, 0.0 * q)


def _ls_phase_case(case, mat, h):
    sc = dict(ndim=case["ndim"], model="spm", gamma=(mat[0], mat[0]), pinf=(mat[1], mat[1]), dx=[h] * case["ndim"],
              bc=[(case["bc"], case["bc"])] * case["ndim"], limiter=False, thinc=False, viscous=False, f64=True)
    weno, sc["recon"] = case["recon"].split("_")
    sc["weno"] = weno
    return sc


def _ls_cut_rhs(c, W, A, dg, nr, qg, phase, h):
    nd = nr.shape[0]
    R = torch.zeros_like(W)
    for d in range(nd):
        F, _ = _flux(c, W, W, c["dx"], d, 0.0)
        a = A[d] if phase == 1 else 1.0 - A[d]
        F = torch.where(a > 0.0, a * F, 0.0 * F)
        m = W.shape[-1 - d]
        R = R - (_win(F, d, 1, m) - _win(F, d, 0, m)) / h
    f = (1.0 if phase == 1 else -1.0) * qg[nd] * dg / h ** nd
    un = sum(qg[e] * nr[e] for e in range(nd))
    add = torch.cat([torch.zeros_like(f)[None], f * nr, (f * un)[None]])
    return R + torch.where(dg > 0.0, add, 0.0 * add)


def _ls_mix(aU, a0, a1, nrm, amix, bc):
    nd = nrm.shape[0]
    shape = a1.shape
    mixing = ((a1 == 0.0) & (a0 > 0.0)) | ((a1 > 0.0) & (a0 == 0.0)) | (a1 < amix)
    coord = torch.meshgrid(*[torch.arange(m, device=a1.device) for m in shape], indexing="ij")
    sg = [torch.sign(nrm[e]).to(torch.int64) for e in range(nd)]
    beta, tgt, aT = [], [], []
    for mask in range(1, 2 ** nd):
        idx, ok = torch.zeros_like(coord[0]), torch.ones_like(mixing)
        w = torch.ones_like(a1)
        for e in reversed(range(nd)):
            k, m = coord[nd - 1 - e], shape[nd - 1 - e]
            if (mask >> e) & 1:
                k = k + sg[e]
                ok = ok & (sg[e] != 0)
                if bc != "periodic":
                    ok = ok & (k >= 0) & (k < m)
                k = k % m
                w = w * nrm[e].abs()
            idx = idx * m + k
        bits = bin(mask).count("1")
        w = w * w if bits == 1 else (torch.pow(w * w, 1.0 / 3.0) if bits == 3 else w)
        t = a1.reshape(-1)[idx]
        beta.append(torch.where(ok, w * t, 0.0 * w))
        tgt.append(idx)
        aT.append(t)
    tot = sum(beta)
    on = mixing & (tot > 0.0)
    out = aU.reshape(aU.shape[0], -1).clone()
    flat = aU.reshape(aU.shape[0], -1)
    own = torch.zeros_like(flat)
    sel = on.reshape(-1).nonzero()[:, 0]
    for b, t, at in zip(beta, tgt, aT):
        bb = b.reshape(-1)[sel] / tot.reshape(-1)[sel]
        ai, ti, a_t = a1.reshape(-1)[sel], t.reshape(-1)[sel], at.reshape(-1)[sel]
        den = ai * bb + a_t
        f = torch.where(bb > 0.0, bb / torch.where(den > 0.0, den, torch.ones_like(den)), 0.0 * bb)
        M = f * (flat[:, ti] * ai - flat[:, sel] * a_t)
        own[:, sel] += M
        out.index_add_(1, ti, -M)
    return (out + own).reshape(aU.shape)


def _ls_advance(case, phi, W1, W2, h, dt):
    bc, nd = case["bc"], case["ndim"]
    cs = [_ls_phase_case(case, m, h) for m in _LS_MAT]
    A, al, dg, nr = _ls_geometry(phi, h, bc)
    aU = [al * _cons(cs[0], W1), (1.0 - al) * _cons(cs[1], W2)]
    W = [W1, W2]
    qg = _ls_extend(_ls_interface(W[0], W[1], al, dg, nr), phi, al, dg, nr, 2, 20, bc)
    for _ in range(case["steps"]):
        U0, phi0 = list(aU), phi
        for stage, (ca, cb) in enumerate(((0.0, 1.0), (0.75, 0.25), (1.0 / 3.0, 2.0 / 3.0))):
            R = [_ls_cut_rhs(cs[k], W[k], A, dg, nr, qg, k + 1, h) for k in range(2)]
            phi = ca * phi0 + cb * (phi + dt * _ls_advect_rhs(phi, qg[:nd], h, bc))
            aU = [ca * U0[k] + cb * (aU[k] + dt * R[k]) for k in range(2)]
            if stage == 2:
                phi = _ls_reinit(phi, h, bc, 10)
            old = al
            A, al, dg, nr = _ls_geometry(phi, h, bc)
            aU = [_ls_mix(aU[0], old, al, nr, 0.6, bc), _ls_mix(aU[1], 1.0 - old, 1.0 - al, -nr, 0.6, bc)]
            for k, a in enumerate((al, 1.0 - al)):
                new = _prim(cs[k], aU[k] / torch.where(a > 0.0, a, torch.ones_like(a)))
                W[k] = torch.where(a > 0.0, new, W[k])
            W = [_ls_extend(W[k], phi, al, dg, nr, k, 10, bc) for k in range(2)]
            qg = _ls_extend(_ls_interface(W[0], W[1], al, dg, nr), phi, al, dg, nr, 2, 20, bc)
    return [phi, aU[0], aU[1], W[0], W[1], qg]


def exact(case, seed):
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    fam = case["family"]
    if fam == "flow":
        W, dx = _field(case, seed)
        c = _solver_case(case, dx)
        st = DT if c["f64"] else torch.float32
        Us = _cons(c, torch.from_numpy(np.ascontiguousarray(W))).to(st).to(dev)
        U = Us.to(DT)
        op = case["op"]
        if op == "step":
            return _advance(c, U, case["steps"])
        dt = _vjp_dt(case, dx)
        if op == "rhs":
            return _rhs(c, U, dt)
        U.requires_grad_(True)
        y = _rhs(c, U, dt) if op == "rhs_vjp" else _rk3(c, U, dt)
        bar = _adjoint_seed(case, seed, Us).to(DT)
        return torch.autograd.grad(y, U, bar)[0]
    if fam == "batch":
        out = []
        for c in _drops(case, seed):
            U = _cons(c, torch.from_numpy(c["W"])).to(DT if c["f64"] else torch.float32).to(DT).to(dev)
            out.append(_advance(c, U, case["steps"]))
        return out
    phi, W1, W2, vel, h, dt = _levelset(case, seed)
    phi, W1, W2, vel = [torch.from_numpy(np.ascontiguousarray(a)).to(dev) for a in (phi, W1, W2, vel)]
    if fam == "ls_step":
        return _ls_advance(case, phi, W1, W2, h, dt)
    bc, dt = case["bc"], 0.3 * h
    p1 = phi + dt * _ls_advect_rhs(phi, vel, h, bc)
    p2 = 0.75 * phi + 0.25 * (p1 + dt * _ls_advect_rhs(p1, vel, h, bc))
    phi = phi / 3.0 + 2.0 / 3.0 * (p2 + dt * _ls_advect_rhs(p2, vel, h, bc))
    phi = _ls_reinit(phi, h, bc, 10)
    A, al, dg, nr = _ls_geometry(phi, h, bc)
    return [phi, torch.cat([a.reshape(-1) for a in A]), al, dg, nr]
