"""The short paths of the level-set kernels against their long ones: the
reinitialisation's float screen (results must be those of evaluating every
cell in double, bit for bit), the geometry's one-sign cells (both kinds of a
grid's cells against the oracle), the extension of fields that are 0 away from
the interface and its two weight paths."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import oracle as orc  # noqa: E402
import paper_2402_05193_gb300 as jxf  # noqa: E402

P, Z, S = orc.PERIODIC, orc.ZEROGRAD, orc.SYMMETRY


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    torch.cuda.set_device(0)


def _phi(ndim, n, h, seed, amp):
    rng = np.random.default_rng(seed)
    ax = np.meshgrid(*[(np.arange(n[e]) + 0.5) * h for e in reversed(range(ndim))], indexing="ij")
    r = np.sqrt(sum((a - 0.5 * a.max()) ** 2 for a in ax))
    phi = 0.3 * min(n) * h - r
    return phi * (1.0 + amp * np.cos(5.0 * phi / (min(n) * h) + rng.uniform(0, 6))) + \
        amp * 0.02 * h * rng.standard_normal(phi.shape)


@pytest.mark.parametrize("h", [1.0 / 64, 1e-5, 3e4])
@pytest.mark.parametrize("amp", [0.0, 0.05, 0.6])
@pytest.mark.parametrize("ndim,n,bc", [(2, [37, 29], [(S, Z), (P, P)]), (3, [21, 17, 13], [(P, P), (Z, S), (S, S)])])
def test_reinit_screen_is_exact(ndim, n, bc, amp, h):
    """Zeroing by the threshold commutes with the screen: R(thr) is R(0)
    where |R(0)| > thr and 0 elsewhere, to the last bit."""
    grid = jxf.ls_grid(ndim, n, h, bc)
    phi = _phi(ndim, n, h, 1, amp)
    phi.flat[5] = 0.0
    p = torch.from_numpy(phi).cuda()
    full, part = torch.zeros_like(p), torch.zeros_like(p)
    jxf.jxf_ls_reinit_rhs(grid, p, p, 0.0, full)  # threshold 0: every cell in double
    for thr in (1e-3, 5e-2, 0.5, 2.0):
        jxf.jxf_ls_reinit_rhs(grid, p, p, thr, part)
        want = torch.where(full.abs() > thr, full, torch.zeros_like(full))
        assert torch.equal(part, want), thr
    ref = orc.ls_reinit_rhs(orc.ls_config(ndim=ndim, n=n, h=h, bc=bc), phi, phi, 5e-2)
    jxf.jxf_ls_reinit_rhs(grid, p, p, 5e-2, part)
    assert np.abs(part.cpu().numpy() - ref).max() < 1e-12


def test_reinit_screen_leaves_odd_values_to_double():
    """Values the float screen cannot hold: huge, infinite and NaN cells give
    what the double evaluation gives, their neighbours too."""
    grid = jxf.ls_grid(2, [40, 24], 1.0 / 40, [(Z, Z)] * 2)
    phi = _phi(2, [40, 24], 1.0 / 40, 2, 0.05)
    phi[3, 4], phi[10, 11], phi[17, 30] = 1e300, np.inf, np.nan
    p = torch.from_numpy(phi).cuda()
    full, part = torch.zeros_like(p), torch.zeros_like(p)
    jxf.jxf_ls_reinit_rhs(grid, p, p, 0.0, full)
    jxf.jxf_ls_reinit_rhs(grid, p, p, 5e-2, part)
    want = torch.where(full.abs() <= 5e-2, torch.zeros_like(full), full)
    assert torch.equal(part.isnan(), want.isnan())
    assert torch.equal(part.nan_to_num(), want.nan_to_num())


@pytest.mark.parametrize("steps", [1, 2, 7, 20])
def test_extension_from_a_band(steps):
    """Fields that are 0 away from the cut cells, odd and even step counts,
    signed zeros and a NaN normal component among the data."""
    n, h, bc = [23, 19, 17], 1.0 / 16, [(P, P), (Z, S), (S, Z)]
    cfg, grid = orc.ls_config(ndim=3, n=n, h=h, bc=bc), jxf.ls_grid(3, n, h, bc)
    phi = _phi(3, n, h, 3, 0.05)
    _, al, dg, nr = orc.ls_geometry(cfg, phi)
    q = np.where((al > 0) & (al < 1), np.random.default_rng(4).uniform(-1, 1, (4,) + phi.shape), 0.0)
    q[:, 0, 0, :3] = -0.0
    ref = orc.ls_extend(cfg, phi, q, 2, steps)
    d = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (phi, al, dg, nr, q)]
    scr = torch.full((4 * phi.size,), 7.0, dtype=torch.float64, device="cuda")
    jxf.jxf_ls_extend(grid, *d, 4, 2, steps, scr)
    assert np.abs(d[4].cpu().numpy() - ref).max() < 1e-13


@pytest.mark.parametrize("ndim,n,centre", [(2, [50, 40], (1, 2)), (2, [256, 9], (255, 4)), (3, [24, 21, 18], (0, 20, 1)),
                                           (3, [17, 64, 5], (8, 33, 2)), (3, [6, 6, 90], (3, 3, 0))])
def test_extension_leaves_out_empty_blocks(ndim, n, centre):
    """A small drop, most blocks of the grid empty and its band reaching others
    along each axis and across the periodic sides: the interface quantities
    that jxf_ls_init extends are those of jxf_ls_interface and the plain
    extension (20 convex combinations: 1e-13 of the largest value)."""
    h, bc, gamma, pinf = 1.0 / 16, [(P, P)] * ndim, (1.4, 1.67), (0.0, 0.3)
    grid = jxf.ls_grid(ndim, n, h, bc)
    dist = []
    for e in range(ndim):
        x = np.abs(np.arange(n[e]) - centre[e] + 0.25)
        dist.append(np.minimum(x, n[e] - x) * h)
    mesh = np.meshgrid(*dist[::-1], indexing="ij")
    phi = 1.6 * h - np.sqrt(sum(m * m for m in mesh))
    rng = np.random.default_rng(5)
    W = [torch.from_numpy(rng.uniform(0.5, 1.5, (ndim + 2,) + phi.shape)).cuda() for _ in range(2)]
    eos = []
    for k in range(2):
        e = jxf.jxf_eos()
        e.model = jxf.JXF_SPM
        e.gamma[0] = e.gamma[1] = gamma[k]
        e.pinf[0] = e.pinf[1] = pinf[k]
        eos.append(e)
    sch = jxf.jxf_scheme()
    sch.recon, sch.precision, sch.weno_eps = jxf.JXF_WENO5JS_CHAR, jxf.JXF_FP64, 1e-6
    d = torch.from_numpy(np.ascontiguousarray(phi)).cuda()
    z = lambda k: torch.zeros((k,) + phi.shape, dtype=torch.float64, device="cuda")
    got = z(ndim + 1)
    work = torch.full((jxf.jxf_ls_step_work(grid),), 3.0, dtype=torch.float64, device="cuda")
    jxf.jxf_ls_init(grid, *eos, sch, d, *W, z(ndim + 2), z(ndim + 2), got, work)
    ap = torch.zeros(jxf.jxf_ls_nface(grid), dtype=torch.float64, device="cuda")
    al, dg, nr, want = z(1)[0], z(1)[0], z(ndim), z(ndim + 1)
    jxf.jxf_ls_geometry(grid, d, ap, al, dg, nr)
    jxf.jxf_ls_interface(grid, *W, gamma, pinf, al, dg, nr, want[:ndim], want[ndim])
    jxf.jxf_ls_extend(grid, d, al, dg, nr, want, ndim + 1, 2, 20, z(ndim + 1))
    assert want.abs().max() > 0.1
    assert (got - want).abs().max() < 1e-13 * want.abs().max()


def _same_with_nans(a, b):
    a, b = a.cpu().numpy(), b.cpu().numpy()
    assert np.isnan(b).any() and np.array_equal(np.isnan(a), np.isnan(b))
    assert np.abs(np.nan_to_num(a) - np.nan_to_num(b)).max() < 1e-13


@pytest.mark.parametrize("steps", [1, 4, 20])
def test_extension_with_a_nan_normal(steps):
    """A NaN normal component in a cell whose values and neighbours are +0: 0
    times NaN is evaluated.  Against the same data with 1e-290 for 0, where
    nothing is left out."""
    n, h, bc = [23, 19, 17], 1.0 / 16, [(P, P), (Z, S), (S, Z)]
    cfg, grid = orc.ls_config(ndim=3, n=n, h=h, bc=bc), jxf.ls_grid(3, n, h, bc)
    phi = _phi(3, n, h, 3, 0.05)
    _, al, dg, nr = orc.ls_geometry(cfg, phi)
    cut = ((al > 0) & (al < 1)) | (dg > 0)
    k = tuple(np.argwhere(~cut & (np.abs(phi) > 3.5 * h))[0])
    nr[(0,) + k] = np.nan
    out = []
    for zero in (0.0, 1e-290):
        q = np.where(cut, np.random.default_rng(4).uniform(-1, 1, (4,) + phi.shape), zero)
        d = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (phi, al, dg, nr, q)]
        jxf.jxf_ls_extend(grid, *d, 4, 2, steps, torch.empty(4 * phi.size, dtype=torch.float64, device="cuda"))
        out.append(d[4])
    _same_with_nans(*out)


@pytest.mark.parametrize("ndim,n,bad", [(2, [50, 40], (30, 25)), (2, [256, 9], (4, 100)), (3, [24, 21, 18], (9, 12, 12))])
def test_empty_blocks_beside_a_nan(ndim, n, bad):
    """A NaN level set in an otherwise empty block: the interface quantities of
    jxf_ls_init, which leave empty blocks out, are NaN where the plain
    extension's are."""
    h, bc, gamma, pinf = 1.0 / 16, [(P, P)] * ndim, (1.4, 1.67), (0.0, 0.3)
    grid = jxf.ls_grid(ndim, n, h, bc)
    mesh = np.meshgrid(*[(np.arange(m) - 4.3) * h for m in n][::-1], indexing="ij")
    phi = 1.6 * h - np.sqrt(sum(m * m for m in mesh))
    phi[tuple(min(b, s - 1) for b, s in zip(bad, phi.shape))] = np.nan
    rng = np.random.default_rng(5)
    W = [torch.from_numpy(rng.uniform(0.5, 1.5, (ndim + 2,) + phi.shape)).cuda() for _ in range(2)]
    eos = []
    for k in range(2):
        e = jxf.jxf_eos()
        e.model = jxf.JXF_SPM
        e.gamma[0] = e.gamma[1] = gamma[k]
        e.pinf[0] = e.pinf[1] = pinf[k]
        eos.append(e)
    sch = jxf.jxf_scheme()
    sch.recon, sch.precision, sch.weno_eps = jxf.JXF_WENO5JS_CHAR, jxf.JXF_FP64, 1e-6
    d = torch.from_numpy(np.ascontiguousarray(phi)).cuda()
    z = lambda k: torch.zeros((k,) + phi.shape, dtype=torch.float64, device="cuda")
    got = z(ndim + 1)
    work = torch.full((jxf.jxf_ls_step_work(grid),), 3.0, dtype=torch.float64, device="cuda")
    jxf.jxf_ls_init(grid, *eos, sch, d, *W, z(ndim + 2), z(ndim + 2), got, work)
    ap = torch.zeros(jxf.jxf_ls_nface(grid), dtype=torch.float64, device="cuda")
    al, dg, nr, want = z(1)[0], z(1)[0], z(ndim), z(ndim + 1)
    jxf.jxf_ls_geometry(grid, d, ap, al, dg, nr)
    jxf.jxf_ls_interface(grid, *W, gamma, pinf, al, dg, nr, want[:ndim], want[ndim])
    jxf.jxf_ls_extend(grid, d, al, dg, nr, want, ndim + 1, 2, 20, z(ndim + 1))
    _same_with_nans(got, want)


@pytest.mark.parametrize("amp", [0.0, 0.05, 0.6])
def test_reinit_screen_is_exact_where_cells_are_gathered(amp):
    """The same above one block per SM, in the kernel that gathers."""
    test_reinit_screen_is_exact(3, [37, 35, 33], [(P, P), (Z, S), (S, S)], amp, 1.0 / 64)
