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
