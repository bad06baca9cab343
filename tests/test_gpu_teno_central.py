"""Double TENO6-A faces that keep every candidate for certain take the linear
six-cell value; the others the full evaluation.  Both against the oracle: from
uniform data over resolved waves to data that drops stencils everywhere, a pure
entropy wave, dimensional data, mirrored walls.
Bar: 1e-13 for one right-hand side as it enters one update, as for the other
right-hand-side cases."""
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


def _check(case):
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


@pytest.mark.parametrize("amp", [0.0, 1e-3, 0.1, 0.45])
@pytest.mark.parametrize("recon", ["char", "comp"])
@pytest.mark.parametrize("ndim,n,bc,visc", [(1, [97], "periodic", 2), (2, [61, 53], "zerograd", 4),
                                            (3, [23, 21, 26], "symmetry", 6), (3, [9, 7, 8], "periodic", 6)])
def test_single_phase(ndim, n, bc, visc, recon, amp):
    _check(dict(wl.smooth_random(ndim, n, "spm", seed=11, recon=recon, bc=bc, amp=amp, viscous=True, mu=1e-2),
                weno="teno6a", visc_order=visc))


@pytest.mark.parametrize("kind", ["entropy wave", "air units"])
def test_cancelling_characteristics(kind):
    case = wl.smooth_random(2, [83, 31], "spm", seed=12, recon="char", amp=0.1)
    W = case["W"].copy()
    if kind == "entropy wave":
        W[1:3] = 0.3
        W[3] = 1.0
    if kind == "air units":
        W[0] *= 1.2
        W[1:3] *= 340.0
        W[3] *= 101325.0
    _check(dict(case, W=np.ascontiguousarray(W), weno="teno6a"))


@pytest.mark.parametrize("recon", ["char", "comp"])
def test_five_equation(recon):
    _check(dict(wl.smooth_random(2, [41, 37], "dim", seed=13, recon=recon, amp=0.02, limiter=True, gamma=(1.4, 1.66),
                                 rho=(1.2, 0.17), p0=1e5, u0=30.0), weno="teno6a"))


@pytest.mark.parametrize("n,axis", [((1170,), 0), ((1170, 5), 0), ((5, 1170), 1)])
@pytest.mark.parametrize("recon", ["comp", "char"])
def test_jumps_between_constant_states(recon, n, axis):
    """Steps of 1e3 to 2e4 in data in physical units (pressure component-wise,
    density where the characteristic variables carry it), up and down, at every
    place of a block of 128 faces: beside flat cells tau6/beta spans float's
    range, and only the flat side may be kept."""
    ndim = len(n)
    J = np.geomspace(1e3, 2e4, 65)
    q = np.full(130, 1e5)
    q[1::2] += J
    q = np.repeat(q, 9).reshape([n[axis] if e == axis else 1 for e in (2, 1, 0)])
    case = wl.smooth_random(ndim, list(n), "spm", seed=1, recon=recon, bc="zerograd", amp=0.0)
    W = np.empty_like(case["W"])
    W[0], W[1:1 + ndim], W[1 + ndim] = 1.2, 3.0, 1e5
    W[0 if recon == "char" else 1 + ndim] = q
    _check(dict(case, W=W, weno="teno6a"))
