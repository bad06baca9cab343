"""The double WENO5 sweeps' two face paths -- nonlinear correction and HLLC
dissipation in float pairs where the stencil is resolved, all double elsewhere
-- against the oracle, on both sides of the criterion and of the range the
pairs cover.  Bar: 1e-13 for one right-hand side as it enters one update, the
bar of the other right-hand-side cases."""
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
    for ndim, n, bc in ((2, [33, 17], "zerograd"), (3, [9, 7, 11], "symmetry")):
        _check(dict(wl.smooth_random(ndim, n, "spm", seed=3, recon=recon, bc=bc, amp=amp, **SCALES[scale]),
                    weno=weno))


@pytest.mark.parametrize("weno", ["js", "z"])
@pytest.mark.parametrize("recon", ["char", "comp"])
@pytest.mark.parametrize("amp", [1e-4, 0.1])
def test_five_equation_stiffened(amp, recon, weno):
    _check(dict(wl.smooth_random(2, [29, 23], "dim", seed=5, recon=recon, amp=amp, limiter=True, gamma=(6.12, 1.4),
                                 pinf=(3.43e8, 0.0), rho=(1000.0, 1.2), p0=1e5, u0=30.0), weno=weno))


def test_resolved_and_unresolved_faces_in_one_warp():
    """A jump in a smooth field: neighbouring faces of a row take both paths,
    at rest (s* = 0) on one side."""
    case = wl.smooth_random(2, [67, 5], "spm", seed=9, recon="char", bc="zerograd", amp=0.02)
    W = case["W"].copy()
    W[:, :, :, 31:] = W[:, :, :, 31:32]
    W[1:3, :, :, 31:] = 0.0
    W[0, :, :, 31:] *= 0.125
    W[3, :, :, 31:] *= 0.1
    _check(dict(case, W=np.ascontiguousarray(W)))
