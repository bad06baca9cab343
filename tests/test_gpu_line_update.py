"""The 1-D stage kernel (faces and update in one block, lane groups sharing a
double face's weights) against the oracle at the edges of its blocks: one
block, its last cell, the first of the next, the last size with lane groups
and the first without.  Two steps: 6 right-hand sides at 1e-13 of an update
each."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import oracle  # noqa: E402
import paper_2402_05193_gb300 as jxf  # noqa: E402
from case_tools import oracle_config, rel_linf  # noqa: E402
from paper_2402_05193_gb300 import workloads as wl  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    torch.cuda.set_device(0)


@pytest.mark.parametrize("bc", ["periodic", "zerograd", "symmetry"])
@pytest.mark.parametrize("model,recon,weno", [("spm", "char", "js"), ("spm", "comp", "z"), ("dim", "char", "js"),
                                              ("spm", "char", "teno6a")])
@pytest.mark.parametrize("n", [3, 15, 16, 31, 32, 63, 127, 128, 254, 255, 2280, 2281, 4712, 4713])
def test_two_steps(n, model, recon, weno, bc):
    kw = dict(rho=(1.2, 0.17), p0=1e5, u0=30.0) if model == "dim" else {}
    case = dict(wl.smooth_random(1, [n], model, seed=n, bc=bc, amp=0.1, recon=recon, limiter=model == "dim", **kw),
                weno=weno)
    c = oracle_config(case)
    U0 = oracle.prim_to_cons(c, case["W"])
    Ur, tr, *_ = oracle.run(c, U0, 2)
    s = jxf.Solver(case, "fp64")
    s.set_primitive(case["W"])
    t = s.step(2)
    U = s.state().cpu().numpy()
    s.close()
    assert abs(t - tr) <= 1e-12 * tr
    assert rel_linf(U, Ur).max() < 1e-12


@pytest.mark.parametrize("prec,tol", [("fp64", 1e-12), ("fp32", 1e-5)])  # float: 6 updates, 30 ulps each
@pytest.mark.parametrize("weno", ["js", "teno6a"])
@pytest.mark.parametrize("order", [2, 4, 6])
@pytest.mark.parametrize("n", [31, 200, 4712, 4713])
def test_viscous_steps(n, order, weno, prec, tol):
    """Every viscous stencil in the stage kernel, with the temperature's three
    buffers, on both sides of the lane-group limit."""
    case = dict(wl.smooth_random(1, [n], "spm", seed=n, bc="zerograd", amp=0.1, recon="char", viscous=True, mu=0.02 / n),
                weno=weno, visc_order=order)
    c = oracle_config(case)
    U0 = oracle.prim_to_cons(c, case["W"])
    Ur, tr, *_ = oracle.run(c, U0, 4)
    s = jxf.Solver(case, prec)
    s.set_primitive(case["W"])
    t = s.step(4)
    U = s.state().cpu().numpy()
    s.close()
    assert abs(t - tr) <= tol * tr
    assert rel_linf(U, Ur).max() < tol


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("kind", ["viscous", "five-equation", "teno6a"])
@pytest.mark.parametrize("n,nblocks,bc", [(48, 2, "periodic"), (96, 3, "zerograd"), (9426, 2, "zerograd")])
def test_blocks_of_a_line(n, nblocks, bc, kind, prec):
    """A 1-D grid in blocks: bit for bit the single grid's, as in two and three
    dimensions (one block of 4713 cells: the whole grid decides on lane groups)."""
    from paper_2402_05193_gb300.decomp import SlabGrid
    if kind == "five-equation":
        case = dict(wl.smooth_random(1, [n], "dim", seed=2, bc=bc, amp=0.1, recon="char", limiter=True, gamma=(1.4, 1.66),
                                     rho=(1.2, 0.17), p0=1e5, u0=30.0), thinc=True)
    else:
        case = dict(wl.smooth_random(1, [n], "spm", seed=2, bc=bc, amp=0.1, recon="char", viscous=True, mu=0.02 / n),
                    weno="teno6a" if kind == "teno6a" else "js", visc_order=6)
    out = []
    for make in (lambda: jxf.Solver(case, prec), lambda: SlabGrid(case, prec, nblocks)):
        s = make()
        s.set_primitive(case["W"])
        s.step(10)
        out.append((s.state().cpu().numpy(),) + tuple(s.stats()[1:]))
        s.close()
    assert np.array_equal(out[0][0], out[1][0])
    assert out[0][1:] == out[1][1:]
