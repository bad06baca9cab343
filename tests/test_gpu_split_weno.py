"""The double WENO5 sweeps' two face paths -- nonlinear correction and HLLC
dissipation in float pairs where the stencil is resolved, all double elsewhere
-- against the oracle, on both sides of the criterion and of the range the
pairs cover, and the reverse sweep's.  Grids above and below the size from
which the choice is made face by face.  Bar: 1e-13 for one right-hand side as
it enters one update, the bar of the other right-hand-side cases."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import oracle  # noqa: E402
import paper_2402_05193_gb300 as jxf  # noqa: E402
from case_tools import momentum_slice, oracle_config, rhs_update_err  # noqa: E402
from paper_2402_05193_gb300 import workloads as wl  # noqa: E402

TOL = 1e-13


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    torch.cuda.set_device(0)


def _check(case, eps=None):
    c = oracle_config(case)
    U = oracle.prim_to_cons(c, case["W"])
    dt = oracle.dt(c, U)
    R_ref, _ = oracle.rhs(c, U, 0.5 * dt)
    s = jxf.Solver(case, "fp64")
    R = s.rhs(torch.from_numpy(U).cuda(), 0.5 * dt).cpu().numpy()
    s.close()
    err = rhs_update_err(R, R_ref, U, dt, momentum_slice(case))
    assert np.isfinite(R).all()
    assert err.max() < TOL, err


SCALES = {"unit": dict(rho=(1.0, 0.5), p0=1.0, u0=0.3), "air": dict(rho=(1.2, 0.17), p0=1e5, u0=100.0),
          "thin": dict(rho=(1e-6, 1e-6), p0=1e-6, u0=0.3)}  # thin: below the pairs' range


@pytest.mark.parametrize("amp", [0.0, 1e-12, 1e-3, 0.1, 0.45])
@pytest.mark.parametrize("recon,weno", [("char", "js"), ("char", "z"), ("comp", "js"), ("comp", "z")])
@pytest.mark.parametrize("scale", list(SCALES))
def test_single_phase(scale, recon, weno, amp):
    for ndim, n, bc in ((2, [33, 17], "zerograd"), (2, [157, 131], "zerograd"), (3, [29, 27, 26], "symmetry")):
        _check(dict(wl.smooth_random(ndim, n, "spm", seed=3, recon=recon, bc=bc, amp=amp, **SCALES[scale]),
                    weno=weno))


@pytest.mark.parametrize("weno", ["js", "z"])
@pytest.mark.parametrize("recon", ["char", "comp"])
@pytest.mark.parametrize("amp", [1e-4, 0.1])
def test_five_equation_stiffened(amp, recon, weno):
    _check(dict(wl.smooth_random(2, [161, 123], "dim", seed=5, recon=recon, amp=amp, limiter=True, gamma=(6.12, 1.4),
                                 pinf=(3.43e8, 0.0), rho=(1000.0, 1.2), p0=1e5, u0=30.0), weno=weno))


def test_resolved_and_unresolved_faces_in_one_warp():
    """A jump in a smooth field: neighbouring faces of a row take both paths,
    at rest (s* = 0) on one side."""
    case = wl.smooth_random(2, [331, 61], "spm", seed=9, recon="char", bc="zerograd", amp=0.02)
    W = case["W"].copy()
    W[:, :, :, 31:] = W[:, :, :, 31:32]
    W[1:3, :, :, 31:] = 0.0
    W[0, :, :, 31:] *= 0.125
    W[3, :, :, 31:] *= 0.1
    _check(dict(case, W=np.ascontiguousarray(W)))


@pytest.mark.parametrize("recon,weno", [("char", "js"), ("char", "z"), ("comp", "js"), ("comp", "z")])
@pytest.mark.parametrize("amp", [0.02, 0.3])
@pytest.mark.parametrize("ndim,n,bc", [(2, [163, 121], "symmetry"), (3, [30, 27, 26], "periodic")])
def test_reverse_sweep_against_the_oracle_tangent(ndim, n, bc, amp, recon, weno):
    """<Ubar, v> = <Rbar, (dR/dU) v> with the oracle's dual-number tangent, for
    random Rbar and v, relative to the sum of the products' magnitudes: every
    term is accurate to about 1e-13 of its own size (the right-hand side's bar)."""
    case = dict(wl.smooth_random(ndim, n, "spm", seed=21, recon=recon, bc=bc, amp=amp), weno=weno)
    c = oracle_config(case)
    U = oracle.prim_to_cons(c, case["W"])
    rng = np.random.default_rng(22)
    v, rbar = rng.standard_normal(U.shape), rng.standard_normal(U.shape)
    _, Rv = oracle.rhs_tangent(c, U, v)
    s = jxf.Solver(case, "fp64")
    g = s.rhs_vjp(torch.from_numpy(U).cuda(), torch.from_numpy(rbar).cuda()).cpu().numpy()
    s.close()
    a, b = float(np.sum(g * v)), float(np.sum(rbar * Rv))
    size = float(np.sum(np.abs(g * v)) + np.sum(np.abs(rbar * Rv)))
    print("<Ubar, v> %.17g, <Rbar, R'v> %.17g, rel %.2e" % (a, b, abs(a - b) / size))
    assert abs(a - b) < 1e-13 * size


def test_level_set_cut_faces_sorted():
    """The level-set sweep's dry, resolved and unresolved faces (sorted within
    each block) against the oracle's cut-cell right-hand side."""
    n, h = [31, 29, 27], 1.0 / 31
    P = orc_bc = (oracle.PERIODIC, oracle.PERIODIC)
    ax = np.meshgrid(*[(np.arange(n[e]) + 0.5) * h for e in (2, 1, 0)], indexing="ij")[::-1]
    phi = 0.3 - np.sqrt(sum((a - 0.5 * a.max()) ** 2 for a in ax))
    w = 0.02 * np.cos(2 * np.pi * (ax[0] / ax[0].max() + ax[1]))
    jump = np.where(ax[2] > 0.7 * ax[2].max(), 3.0, 1.0)
    W = np.stack([(1.0 + w) * jump, 0.3 + w, -0.2 * w, 0.1 + 0 * w, (1.0 + w) * jump])
    cfg = oracle.make_config(ndim=3, n=n, dx=[h] * 3, bc=[orc_bc] * 3, gamma=(1.4, 1.4), recon=oracle.CHAR)
    lcfg = oracle.ls_config(ndim=3, n=n, h=h, bc=[P] * 3)
    ap, al, dg, nr = oracle.ls_geometry(lcfg, phi)
    ug, pg = np.zeros((3,) + phi.shape), np.where(dg > 0, 1.0, 0.0)
    grid = jxf.ls_grid(3, n, h, [(jxf.JXF_BC_PERIODIC,) * 2] * 3)
    eos, sch = jxf.jxf_eos(), jxf.jxf_scheme()
    eos.gamma[0] = eos.gamma[1] = 1.4
    sch.recon, sch.weno_eps = jxf.JXF_WENO5JS_CHAR, 1e-6
    d = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (ap, dg, nr, W, ug, pg)]
    dU = torch.zeros(W.shape, dtype=torch.float64, device="cuda")
    scr = torch.zeros(5 * jxf.jxf_ls_nface(grid), dtype=torch.float64, device="cuda")
    for phase in (1, 2):
        ref = oracle.ls_cut_rhs(cfg, phi, W, phase, ug, pg)
        jxf.jxf_ls_cut_rhs(grid, eos, sch, d[0], d[1], d[2], d[3], phase, d[4], d[5], dU, scr)
        err = np.abs(dU.cpu().numpy() - ref).max() / np.abs(ref).max()
        assert err < 1e-13, (phase, err)


def _bump(weno, recon, weno_eps):
    """Parabolic bumps with a small step at their rim in an otherwise exactly
    uniform state: differences are 0 or well above rounding."""
    case = wl.smooth_random(2, [157, 131], "spm", seed=4, recon=recon, bc="periodic", amp=0.0)
    W = case["W"].copy()
    for v, (cx, cy, a) in enumerate(((40, 30, 0.02), (90, 70, 0.01), (60, 95, -0.01), (110, 40, 0.02))):
        y, x = np.meshgrid(np.arange(131) - cy, np.arange(157) - cx, indexing="ij")
        r2 = (x * x + y * y) / 400.0
        W[v, 0] += np.where(r2 < 1.0, a * (1.05 - r2), 0.0)
    return dict(case, W=W, weno=weno, weno_eps=weno_eps)


@pytest.mark.parametrize("weno_eps", [1e-12, 1e-22, 1e-40, 1e-60])
@pytest.mark.parametrize("recon,weno", [("char", "js"), ("char", "z"), ("comp", "js"), ("comp", "z")])
def test_small_weno_eps(recon, weno, weno_eps):
    """A weight parameter near or below float's range, forward and reverse, in
    uniform regions (indicators 0) as well."""
    case = _bump(weno, recon, weno_eps)
    c = oracle_config(case, weno_eps=weno_eps)
    U = oracle.prim_to_cons(c, case["W"])
    dt = oracle.dt(c, U)
    R_ref, _ = oracle.rhs(c, U, 0.5 * dt)
    rng = np.random.default_rng(23)
    v, rbar = rng.standard_normal(U.shape), rng.standard_normal(U.shape)
    _, Rv = oracle.rhs_tangent(c, U, v)
    s = jxf.Solver(case, "fp64")
    R = s.rhs(torch.from_numpy(U).cuda(), 0.5 * dt).cpu().numpy()
    g = s.rhs_vjp(torch.from_numpy(U).cuda(), torch.from_numpy(rbar).cuda()).cpu().numpy()
    s.close()
    err = rhs_update_err(R, R_ref, U, dt, momentum_slice(case))
    assert np.isfinite(R).all()
    assert err.max() < TOL, err
    # beside uniform cells the weights' derivatives cancel over 1/weno_eps: below
    # 1e-12 the oracle's own tangent loses more than the bar and WENO5-Z's
    # all-double reverse is large itself; the size of Jiang-Shu's is left
    assert np.isfinite(g).all()
    if weno == "js":
        assert np.abs(g).max() < 1e8
    a, b = float(np.sum(g * v)), float(np.sum(rbar * Rv))
    if weno_eps >= 1e-12:
        assert abs(a - b) < 1e-13 * float(np.sum(np.abs(g * v)) + np.sum(np.abs(rbar * Rv)))


def test_trace_partial_density_and_volume_fraction():
    """A rough trace gas carried at the speed of sound: partial density and
    volume fraction, 1e-4 of the mixture's, are accurate to their own size.  Bar
    of one update: 8 roundings of 2^-53 in each of two faces' fluxes and in the
    oracle's, times dt u/dx <= 0.2."""
    case = wl.smooth_random(2, [161, 141], "dim", seed=5, recon="comp", amp=0.02, gamma=(1.4, 1.66), rho=(1.0, 1.0))
    W = case["W"].copy()
    a = 1e-4 * (1.0 + 0.5 * np.random.default_rng(7).uniform(-1, 1, W.shape[1:]))
    W[0], W[1], W[5], W[2], W[3] = a, 1.0 - a, a, 1.0 + W[2] - 0.3, 0.3
    for recon in ("comp", "char"):
        c = oracle_config(dict(case, W=W, recon=recon))
        U = oracle.prim_to_cons(c, W)
        dt = oracle.dt(c, U)
        ref, _ = oracle.rhs(c, U, 0.5 * dt)
        s = jxf.Solver(dict(case, W=W, recon=recon), "fp64")
        R = s.rhs(torch.from_numpy(U).cuda(), 0.5 * dt).cpu().numpy()
        s.close()
        err = rhs_update_err(R, ref, U, dt)
        print(recon, err)
        assert err[[0, 5]].max() < 8 * 2 * 2 * 2.0 ** -53 * 0.1


@pytest.mark.parametrize("recon", ["char", "comp"])
@pytest.mark.parametrize("kind", ["rough", "graded", "wave"])
def test_small_transverse_velocity(kind, recon):
    """A transverse velocity of 1e-3 carried by a uniform flow near the speed of
    sound, constant along y so that no pressure enters its momentum: accurate to
    its own size.  Bar of one update as above with dt u/dx <= 0.15."""
    case = wl.smooth_random(2, [331, 61], "spm", seed=5, recon=recon, amp=0.0)
    rng = np.random.default_rng(8)
    x = np.arange(331)
    v = {"rough": rng.standard_normal(331), "graded": 1.0 + 0.2 * rng.uniform(0, 1, 331) ** 4 * rng.standard_normal(331),
         "wave": np.sin(2 * np.pi * (x + 0.37) / 331)}[kind]
    W = case["W"].copy()
    W[0], W[1], W[2], W[3] = 1.0, 1.0, 1e-3 * v, 1.0
    c = oracle_config(dict(case, W=W))
    U = oracle.prim_to_cons(c, W)
    dt = oracle.dt(c, U)
    ref, _ = oracle.rhs(c, U, 0.5 * dt)
    s = jxf.Solver(dict(case, W=W), "fp64")
    R = s.rhs(torch.from_numpy(U).cuda(), 0.5 * dt).cpu().numpy()
    s.close()
    err = rhs_update_err(R, ref, U, dt)
    print(kind, recon, err)
    assert err[2] < 8 * 2 * 2 * 2.0 ** -53 * 0.15


@pytest.mark.parametrize("recon", ["char", "comp"])
@pytest.mark.parametrize("weno", ["js", "z"])
def test_reverse_sweep_of_uniform_supersonic_flow(weno, recon):
    """At a uniform state, supersonic along both axes, the faces are the
    fifth-order upwind values (2, -13, 47, 27, -3)/60: the reverse sweep in
    closed form (extended precision).  In the mean 1e-15 of the mean: about 8
    roundings of 2^-53."""
    n, dx, g, w = [157, 131], [1.0 / 157, 1.0 / 131], 1.4, (1.0, 2.5, 2.2, 1.0)
    case = dict(wl.smooth_random(2, n, "spm", seed=1, recon=recon, amp=0.0), weno=weno)
    W = np.empty_like(case["W"])
    for v in range(4):
        W[v] = w[v]
    U = oracle.prim_to_cons(oracle_config(case), W)
    rbar = np.random.default_rng(3).standard_normal(U.shape)
    s = jxf.Solver(case, "fp64")
    got = s.rhs_vjp(torch.from_numpy(U).cuda(), torch.from_numpy(rbar).cuda()).cpu().numpy()
    s.close()
    L = np.longdouble
    r, mu, mv, E = (L(U[v].flat[0]) for v in range(4))
    u, v = mu / r, mv / r
    p = (L(g) - 1) * (E - r * (u * u + v * v) / 2)
    h = L(g) / (L(g) - 1)
    ke = (u * u + v * v) / 2
    # dF/dW for the x and y fluxes, dW/dU
    A = [np.array([[u, r, 0, 0], [u * u, 2 * r * u, 0, 1], [u * v, r * v, r * u, 0],
                   [u * ke, h * p + r * ke + r * u * u, r * u * v, h * u]], L),
         np.array([[v, 0, r, 0], [u * v, r * v, r * u, 0], [v * v, 0, 2 * r * v, 1],
                   [v * ke, r * u * v, h * p + r * ke + r * v * v, h * v]], L)]
    k = L(g) - 1
    B = np.array([[1, 0, 0, 0], [-u / r, 1 / r, 0, 0], [-v / r, 0, 1 / r, 0], [k * ke, -k * u, -k * v, k]], L)
    coef = [L(c) / 60 for c in (2, -13, 47, 27, -3)]  # cells i - 2 .. i + 2 of face i + 1/2
    rb, Wb = rbar[:, 0].astype(L), np.zeros((4,) + rbar.shape[2:], L)
    for d, axis in ((0, 2), (1, 1)):
        Fb = (np.roll(rb, -1, axis) - rb) / L(dx[d])  # of face i + 1/2
        for m, c in zip(range(-2, 3), coef):
            Wb += c * np.einsum("fw,fyx->wyx", A[d], np.roll(Fb, m, axis))
    ref = np.einsum("wu,wyx->uyx", B, Wb)
    err = np.abs(got[:, 0] - ref).mean(axis=(1, 2)) / np.abs(ref).mean(axis=(1, 2))
    print(weno, recon, err)
    assert err.max() < 1e-15


@pytest.mark.parametrize("recon,weno", [("char", "js"), ("comp", "z")])
@pytest.mark.parametrize("model,n", [("spm", (138, 139)), ("spm", (139, 140)), ("spm", (33, 34, 33)), ("spm", (36, 34, 32)),
                                     ("dim", (138, 139)), ("dim", (139, 140)), ("dim", (46, 45, 45)), ("dim", (47, 46, 45))])
def test_sizes_beside_the_rule(model, n, recon, weno):
    """Grids below and above the sizes from which faces choose for themselves."""
    kw = dict(gamma=(1.4, 1.66), rho=(1.2, 0.17), p0=1e5, u0=30.0, limiter=True) if model == "dim" else {}
    _check(dict(wl.smooth_random(len(n), list(n), model, seed=6, recon=recon, amp=0.02, **kw), weno=weno))


@pytest.mark.parametrize("recon,weno", [("char", "js"), ("comp", "z")])
def test_reverse_sweep_3d_above_the_rule(recon, weno):
    """As test_reverse_sweep_against_the_oracle_tangent, on a 3-D grid whose
    faces choose for themselves."""
    test_reverse_sweep_against_the_oracle_tangent(3, [36, 34, 32], "periodic", 0.02, recon, weno)
