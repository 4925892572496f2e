"""Kernels at the sizes where their tiling can go wrong (edges of tiles, remainders, the smallest and
largest classes), against the oracle or the library's general path.  Each tolerance is derived in
its test's docstring."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import mesh as om


@pytest.fixture(scope="module")
def mto():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1811_09821_gb300 as m
    from paper_1811_09821_gb300 import _build
    _build.build()
    m.load_library()
    return m


def handle(mto, nx, ny, p, d, hx=1.0, hy=1.0):
    h = mto.Handle(0)
    h.setup(nx, ny, np.broadcast_to(np.asarray(p, np.int32), nx * ny), np.broadcast_to(np.asarray(d, np.int32), nx * ny),
            hx, hy)
    return h


@pytest.mark.parametrize("nx,ny", [(1, 1), (43, 3)])   # 1 and 129 elements: one row, one past a tile of 128
@pytest.mark.parametrize("p", [1, 2, 3, 4, 5, 6])
@pytest.mark.parametrize("d", [1, 4, 5, 8])            # K = 1, 16, 25 (padded to 32) and 64 subcells
def test_tensor_build_edges(mto, nx, ny, p, d):
    """The sliced tensor-core build against the FP64 CUDA-core build: the dropped levels weigh below
    2^-51 of the element's scale and the 64-term FP64 sums below 64 x 2^-53, so 1e-14 of the element's
    largest entry covers both; the split pair is fl32(K) and fl32(K - hi) of the stored FP64
    entries bit for bit, also for moduli of 1e-9 and 1e-24 and for exact zeros."""
    h = handle(mto, nx, ny, p, d)
    rng = np.random.default_rng(100 * p + d)
    rho = rng.uniform(0.0, 1.0, h.design_len)
    rho[rng.uniform(size=len(rho)) < 0.4] = 0.0
    rho[-d * d:] = rng.choice([0.0, 1e-8], d * d)
    rho[:d * d] = 1.0
    r = torch.tensor(rho, device="cuda")
    mat = mto.material(1.0, 0.0 if d == 5 else 1e-9, 0.3, 3.0)
    es = sorted({0, 1, 126, 127, 128} & set(range(nx * ny)))
    h.set_build_path(mto.BUILD_SIMT)
    h.build_elements(r, mat, mto.MTO_FP64)
    want = {e: h.element_matrix(e, p) for e in es}
    h.set_build_path(mto.BUILD_TENSOR)
    h.build_elements(r, mat, mto.MTO_MIXED)
    for e in es:
        got = h.element_matrix(e, p)
        assert np.abs(got - want[e]).max() <= 1e-14 * np.abs(want[e]).max(), e
        hi, lo = h.element_matrix_split(e, p)
        np.testing.assert_array_equal(hi, got.astype(np.float32))
        np.testing.assert_array_equal(lo, (got - hi.astype(np.float64)).astype(np.float32))
    h.close()


@pytest.mark.parametrize("nx,ny,d", [(1, 1, 1), (33, 1, 3), (11, 9, 8), (7, 5, 16), (45, 23, 0)])
def test_density_indicator_and_selection_edges(mto, nx, ny, d):
    """Gamma^d in cell order is the serial sum: bit-equal to the oracle's cell loop (same operations,
    same order) apart from a division by a power of two, which is exact; ragged warps, counts from 1 to
    256 cells, mixed counts (d = 0).  The map update then equals the oracle's on those values and on
    Kelly values full of ties (the stable index tie-break), for several ranks."""
    from oracle import indicators as oi
    rng = np.random.default_rng(nx * 100 + ny)
    nel = nx * ny
    dm = rng.choice([1, 2, 3, 8, 16], nel) if d == 0 else np.full(nel, d)
    p = rng.integers(1, 4, nel)
    h = handle(mto, nx, ny, p, dm)
    m = om.DPMesh(nx, ny, p, dm)
    rho = rng.uniform(0.0, 1.0, h.design_len)
    rho[rng.uniform(size=len(rho)) < 0.3] = rng.choice([0.0, 0.5, 1.0])
    r = torch.tensor(rho, device="cuda")
    mat = mto.material()
    h.set_supports(h.side_dofs(0))
    h.build_elements(r, mat)
    u = torch.tensor(rng.standard_normal(h.ndof), device="cuda")
    for cycle in (1, 3):
        ind = h.indicator(u, r, mat, mto.IndicatorOpts.paper(cycle))
        want = oi.gamma_d(m, rho, cycle)
        np.testing.assert_allclose(ind["gamma_d"].cpu().numpy(), want, rtol=0, atol=1e-15)
        np.testing.assert_allclose(ind["gamma_a"].cpu().numpy(), oi.kelly(m, u.cpu().numpy()), rtol=1e-9, atol=0)
    ga = rng.integers(0, 4, nel).astype(float)          # ties
    gd = want
    eq = rng.uniform(0.0, 1.0, nel)
    for fr, fc in ((0.1, 0.05), (0.5, 0.4), (1.0, 0.0), (0.0, 0.9)):
        o = mto.IndicatorOpts.paper(1)
        o.frac_a_refine, o.frac_a_coarsen = fr, fc
        got = h.map_update(*(torch.tensor(v, device="cuda") for v in (ga, gd, eq)), o)
        pn, dn, th = oi.map_update(nx, ny, p, ga, gd, eq, frac_a_refine=fr, frac_a_coarsen=fc)[:3]
        for a, b in zip(got, (pn, dn, th)):
            np.testing.assert_array_equal(a.cpu().numpy(), b)
    h.close()


@pytest.mark.parametrize("nx,ny", [(1, 1), (13, 5)])
@pytest.mark.parametrize("p", [1, 2, 3, 4, 5, 6])
@pytest.mark.parametrize("d", [1, 2, 3, 8, 16])
def test_sensitivity_edges(mto, nx, ny, p, d):
    """FP64 sensitivities (self-adjoint and bilinear) and the energy form against the oracle's dense
    quadratic forms u^T K0_s u, on one element and ragged blocks, non-square elements: each w_s comes from
    sums of magnitudes below 64 x the element's largest (products of the grid's energy densities with
    integrated Lagrange polynomials whose absolute sums stay below 8 per axis), so 1e-12 of the largest
    value of the mesh bounds the rounding of both sides by two orders."""
    from oracle import sensitivity as ose
    h = handle(mto, nx, ny, p, d, 1.0, 0.5)
    m = om.DPMesh(nx, ny, np.full(nx * ny, p), np.full(nx * ny, d), 1.0, 0.5)
    rng = np.random.default_rng(10 * p + d)
    rho = rng.uniform(0.0, 1.0, h.design_len)
    u, v, f = (rng.standard_normal(h.ndof) for _ in range(3))
    T = lambda a: torch.tensor(a, device="cuda")
    for q in (3.0, 2.5):
        mat = mto.material(1.0, 1e-9, 0.3, q)
        dc, dv = T(np.zeros(h.design_len)), T(np.zeros(h.design_len))
        C = h.sensitivity(T(u), T(f), T(rho), mat, dc)
        assert abs(C - f @ u) <= 1e-12 * np.abs(f) @ np.abs(u)
        want = ose.sensitivity(m, u, rho, q=q)
        assert np.abs(dc.cpu().numpy() - want).max() <= 1e-12 * np.abs(want).max()
        # bilinear form by polarisation of the quadratic one
        h.sensitivity_adjoint(T(u), T(v), T(rho), mat, dv)
        pol = 0.25 * (ose.sensitivity(m, u + v, rho, q=q) - ose.sensitivity(m, u - v, rho, q=q))
        scale = max(np.abs(ose.sensitivity(m, u + v, rho, q=q)).max(), np.abs(ose.sensitivity(m, u - v, rho, q=q)).max())
        assert np.abs(dv.cpu().numpy() - pol).max() <= 1e-12 * scale
        e = ose.energy_split(m, u, rho, q=q)
        assert abs(h.compliance_energy(T(u), T(f), T(rho), mat) - (2.0 * f @ u - e)) <= 1e-12 * (abs(e) + 2 * np.abs(f) @ np.abs(u))
    h.close()


@pytest.mark.parametrize("nx,ny", [(1, 1), (12, 7), (3, 11)])
@pytest.mark.parametrize("d", [1, 3, 5, 8, 16, 0, -1])   # 0, -1: mixed counts (two maps)
@pytest.mark.parametrize("R,hy", [(0.05, 1.0), (0.3, 1.0), (1.0, 0.5), (1.9, 0.5), (4.0, 1.0)])
def test_filter_edges(mto, nx, ny, d, R, hy):
    """The filter's fine-grid stencil (one design count) and its mixed path against the oracle's sparse
    rows: stencils inside, across and wider than the mesh, non-square elements, radii from below one
    subcell to the largest of four elements.  The oracle's subcell centres are rounded at up to 12
    elements (12 x 2^-53), a distance to 8 of those units, a weight of mean R / 3 to 24 / R of them: 4e-14 /
    min(R, 1) covers both sides' rounding with the sums."""
    from oracle import filter as ofl
    if R > 4.0 * min(1.0, hy) or (R > 2.0 and nx > 3 and d in (16, -1)):   # the latter: 10^8 pairs in the oracle
        R = 2.0
    rng = np.random.default_rng(3 + nx)
    nel = nx * ny
    dm = np.full(nel, d) if d > 0 else rng.choice([1, 2, 4, 8] if d == 0 else [1, 3, 7, 16], nel)
    h = handle(mto, nx, ny, 1, dm, 1.0, hy)
    m = om.DPMesh(nx, ny, np.full(nel, 1), dm, 1.0, hy)
    x, g = rng.uniform(size=m.design_len), rng.standard_normal(m.design_len)
    xt, gt = torch.tensor(x, device="cuda"), torch.tensor(g, device="cuda")
    out = torch.empty_like(xt)
    tol = 4e-14 / min(R, 1.0)
    for _ in range(2):
        h.filter(xt, out, R)
        want = ofl.density_filter(m, x, R)
        assert np.abs(out.cpu().numpy() - want).max() <= tol * np.abs(want).max()
        h.filter_adjoint(gt, out, R)
        want = ofl.density_filter_adjoint(m, g, R)
        assert np.abs(out.cpu().numpy() - want).max() <= tol * np.abs(want).max()
    h.close()


@pytest.mark.parametrize("nx,ny", [(1, 1), (1, 9), (9, 1), (2, 1), (31, 31), (500, 1), (3, 200), (5, 4), (40, 23)])
def test_coarsest_inverse_edges(mto, nx, ny):
    """On a Q1 mesh of at most 2048 vertex DOFs the coarsest level is the operator itself, so a V-cycle
    with its exact inverse solves the system and the FP64 PCG takes a few iterations (the FP32 cycle's
    vectors are not checked here: they leave kappa 2^-24 a cycle).  The solution is checked by
    its backward error, which does not depend on the conditioning (a slender cantilever's error in u is
    kappa eps on either side, kappa ~ 1e11 for 500 x 1): every free row's residual with the oracle's K within
    the asked 1e-11 of |f| and 64 eps of that row of |K||u| (18 products and the rounding of K and u).  Lines
    along either axis, one element, two lines, 64 DOFs a line, supported DOFs."""
    from oracle import solve as osv
    rng = np.random.default_rng(nx + 7 * ny)
    h = handle(mto, nx, ny, 1, 2)
    m = om.DPMesh(nx, ny, np.full(nx * ny, 1), np.full(nx * ny, 2))
    rho = rng.uniform(0.1, 1.0, h.design_len)
    fixed, f = mto.load_case(h, "cantilever")
    h.set_supports(fixed)
    K = osv.assemble(m, osv.element_matrices(m, rho, 1.0, 1e-9, 0.3, 3.0))
    free = np.setdiff1d(np.arange(h.ndof), fixed)
    fn = f.cpu().numpy()
    h.build_elements(torch.tensor(rho, device="cuda"), mto.material(), mto.MTO_FP64)
    u = torch.zeros(h.ndof, dtype=torch.float64, device="cuda")
    it, _ = h.solve(f, u, precision=mto.MTO_FP64, rtol=1e-11, precond=mto.PREC_MG, check_every=2, max_iter=200,
                    max_outer=4, raise_on_noconv=False)
    assert it <= 8, it
    un = u.cpu().numpy()
    assert np.all(un[fixed] == 0.0)
    r = np.abs(fn - K @ un)[free]
    assert np.all(r <= 1e-11 * np.linalg.norm(fn) + 64 * 2.0 ** -52 * (abs(K) @ np.abs(un))[free]), r.max()
    h.close()


@pytest.mark.parametrize("nx,ny", [(1, 1), (43, 3)])
@pytest.mark.parametrize("p", [1, 2, 3, 4, 5, 6])
@pytest.mark.parametrize("d", [1, 3, 8, 9])   # the last: more than 64 subcells, summed in the kernel
def test_qr_error_edges(mto, nx, ny, p, d):
    """The QR indicator with order p + 1 matrices formed on the tensor cores (one element, one past a
    tile of 128) and summed in the kernel, against the oracle's dense Cholesky: eps = 1 - J_p / J_(p+1) is
    determined to kappa eps of the pinned element problem, kappa < 1e7 for densities of 0.3 to 1 (modulus
    contrast 40), so 1e-8; the two paths agree with each other to the same bound."""
    from oracle import indicators as oi
    h = handle(mto, nx, ny, p, d)
    m = om.DPMesh(nx, ny, np.full(nx * ny, p), np.full(nx * ny, d))
    rng = np.random.default_rng(p * 31 + d)
    rho = rng.uniform(0.3, 1.0, h.design_len)
    u = rng.standard_normal(h.ndof)
    T = lambda a: torch.tensor(a, device="cuda")
    mat = mto.material()
    h.set_supports(h.side_dofs(0))
    h.build_elements(T(rho), mat)
    got = h.indicator(T(u), T(rho), mat, maps=False)["eps_qr"].cpu().numpy()
    h.set_build_path(mto.BUILD_SIMT)
    ref = h.indicator(T(u), T(rho), mat, maps=False)["eps_qr"].cpu().numpy()
    assert np.abs(got - ref).max() <= 1e-8
    for e in sorted({0, 1, 127, 128} & set(range(nx * ny))):
        want = oi.qr_error_element(p, d, rho[m.design_off[e]:m.design_off[e + 1]], m.gather(e, u), 1.0, 1e-9, 0.3, 3.0)
        assert abs(got[e] - want) <= 1e-8, (e, got[e], want)
    h.close()


@pytest.mark.parametrize("nx,ny,d", [(1, 1, 1), (2, 1, 3), (16, 16, 4), (32, 33, 2), (150, 70, 8), (61, 47, 0)])
@pytest.mark.parametrize("kind", ["late", "uniform", "flat", "void", "unreachable"])
def test_oc_update_edges(mto, nx, ny, d, kind):
    """The OC update that settles values as its interval shrinks (and the one-block path of small designs)
    against the oracle's plain bisection over every value: the same midpoints and the same tests, so
    lambda agrees to the interval's relative width 1e-10 (the volumes' rounding can turn a test only where
    they differ from the target by less than n 2^-53) and the design to 1e-9.  Designs: sensitivities over
    many decades, one value everywhere, steps (many equal breakpoints), no sensitivity at all (the
    interval halves towards 0), and a volume no design within the move limit reaches."""
    from oracle import oc as ooc
    rng = np.random.default_rng(nx + d)
    nel = nx * ny
    dm = np.full(nel, d) if d else rng.choice([1, 2, 4, 8, 5], nel)
    h = handle(mto, nx, ny, 1, dm, 1.0, 0.5 if d == 2 else 1.0)
    n = h.design_len
    rho = rng.uniform(0.0, 1.0, n)
    dc = -np.exp(3.0 * rng.standard_normal(n)) * rho ** 2
    vol = 0.9 * rho.mean() + 0.05
    if kind == "uniform":
        rho[:], dc[:], vol = 0.4, -2.0, 0.4
    if kind == "flat":
        rho, dc = np.round(rho, 1), np.round(dc) - 1.0   # (all zero is "void": the oracle cannot take it)
    if kind == "void":
        dc[:] = 0.0
    if kind == "unreachable":
        vol = 1.0
    m = om.DPMesh(nx, ny, np.full(nel, 1), dm, h.hx, h.hy)
    dv = ooc.subcell_areas(m)
    for eta in (0.5, 0.7):
        out = torch.zeros(n, dtype=torch.float64, device="cuda")
        lam = h.oc_update(torch.tensor(rho, device="cuda"), torch.tensor(dc, device="cuda"), vol, out, eta=eta)
        if kind in ("void", "unreachable"):   # the oracle's loop has no limit of steps there: its design in closed form
            lo, hi = np.maximum(0.0, rho - 0.2), np.minimum(1.0, rho + 0.2)
            want = lo if kind == "void" else np.where(dc < 0.0, hi, lo)
            assert 0.0 < lam < 1e-28
        else:
            want, wl = ooc.oc_update(rho, dc, dv, vol * nel * h.hx * h.hy, eta=eta)
            assert abs(lam - wl) <= 4e-10 * wl
        np.testing.assert_allclose(out.cpu().numpy(), want, rtol=1e-9, atol=1e-12)
    h.close()


@pytest.mark.parametrize("orders", [(1, 1), (1, 2), (2, 3), (1, 4), (4, 5), (3, 6), (1, 2, 3, 4, 5, 6)])
@pytest.mark.parametrize("nx,ny", [(2, 1), (7, 5)])
def test_assembled_diagonal_edges(mto, nx, ny, orders):
    """The assembled diagonal D, read through the scaled norm of the start vector's residual
    (sqrt(r^T D^-1 r / f^T D^-1 f), accepted before the first iteration), against D_i = e_i^T K e_i of the
    FP64 operator, on meshes with and without hanging nodes.  Both sum the same up to a few hundred FP64
    products of entries and weights of order 1 (void at 0.3^3 of solid), so 1e-13 each, and r = f - K u
    of random vectors has no cancellation: 1e-10."""
    rng = np.random.default_rng(nx * 100 + sum(orders))
    p = rng.permutation(np.resize(np.asarray(orders, np.int32), nx * ny))
    h = handle(mto, nx, ny, p, 3)
    T = lambda a: torch.tensor(a, device="cuda")
    fixed = np.asarray(h.side_dofs(0))
    h.set_supports(h.side_dofs(0))
    h.build_elements(T(rng.uniform(0.3, 1.0, h.design_len)), mto.material())
    free = np.setdiff1d(np.arange(h.ndof), fixed)
    D = np.zeros(h.ndof)
    x, y = torch.zeros(h.ndof, dtype=torch.float64, device="cuda"), torch.empty(h.ndof, dtype=torch.float64, device="cuda")
    for i in free:
        x.zero_()
        x[i] = 1.0
        h.apply(x, y)
        D[i] = y[i].item()
    f, u = np.zeros(h.ndof), np.zeros(h.ndof)
    f[free], u[free] = rng.standard_normal(free.size), rng.standard_normal(free.size)
    uT = T(u)
    h.apply(uT, y)
    r = f - y.cpu().numpy()
    want = np.sqrt((r[free] ** 2 / D[free]).sum() / (f[free] ** 2 / D[free]).sum())
    it, got = h.solve(T(f), uT, rtol=1e6, warm_start=True, norm=mto.NORM_JACOBI, precond=mto.PREC_JACOBI)
    assert it == 0
    assert abs(got - want) <= 1e-10 * want
    h.close()
