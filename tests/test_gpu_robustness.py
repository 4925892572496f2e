"""Inputs, sizes and conditions off the usual path: non-finite and negative values, small subcell
energies, failed allocations, several threads.  Each tolerance is derived in its test's docstring."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

T = lambda a: torch.tensor(a, device="cuda")


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


@pytest.mark.parametrize("d", [1, 3, 8, 9])   # the last: more than 64 subcells, the FP64 CUDA-core kernel
@pytest.mark.parametrize("bad", [float("nan"), float("inf"), -0.5, -0.9])
def test_build_of_nonfinite_and_negative_moduli(mto, d, bad):
    """One density that is not a number, infinite or negative, in the second tile of 128 elements or before
    it: the tensor-core build carries it as the FP64 sums do (negative moduli to the 1e-14 of the
    element's largest entry of test_tensor_build_edges), its neighbours keep their bits, the split pair
    follows, and a solve reports MTO_ENAN."""
    nx, ny, p = 43, 3, 2
    rng = np.random.default_rng(d)
    mat = mto.material()
    for e in (64, 128):
        h = handle(mto, nx, ny, p, d)
        rho = rng.uniform(0.2, 1.0, h.design_len)
        fixed, f = mto.load_case(h, "cantilever")
        h.set_supports(fixed)
        h.build_elements(T(rho), mat, mto.MTO_MIXED)
        clean = h.element_matrix(e - 1, p)
        rho[e * d * d] = bad
        h.set_build_path(mto.BUILD_SIMT)
        h.build_elements(T(rho), mat, mto.MTO_FP64)
        want = h.element_matrix(e, p)
        h.set_build_path(mto.BUILD_TENSOR)
        h.build_elements(T(rho), mat, mto.MTO_MIXED)
        got = h.element_matrix(e, p)
        hi, lo = h.element_matrix_split(e, p)
        np.testing.assert_array_equal(h.element_matrix(e - 1, p), clean)
        if np.isfinite(bad):
            assert np.abs(got - want).max() <= 1e-14 * np.abs(want).max()
            np.testing.assert_array_equal(hi, got.astype(np.float32))
            np.testing.assert_array_equal(lo, (got - hi.astype(np.float64)).astype(np.float32))
        else:
            assert not np.isfinite(want).any() and not np.isfinite(got).any() and not np.isfinite(hi).any()
            u = torch.zeros(h.ndof, dtype=torch.float64, device="cuda")
            for pc in (mto.PREC_JACOBI, mto.PREC_SCHWARZ, mto.PREC_MG):
                with pytest.raises(mto.MTOError) as ei:
                    h.solve(f, u, precision=mto.MTO_MIXED, precond=pc, max_iter=50)
                assert ei.value.status == 5
        h.close()


@pytest.mark.parametrize("d", [1, 3, 8, 9])
@pytest.mark.parametrize("bad", [float("nan"), float("inf"), -0.1])
def test_qr_error_of_nonfinite_and_negative_densities(mto, d, bad):
    """The QR indicator of an element with such a density: as the sums in the kernel give it (a modulus of
    -1e-3 beside moduli above 0.125 leaves kappa of the pinned problem below 1e5: 1e-9 between the paths), the
    other elements keep their bits."""
    nx, ny, p, e = 43, 3, 2, 64
    h = handle(mto, nx, ny, p, d)
    rng = np.random.default_rng(d)
    rho = rng.uniform(0.5, 1.0, h.design_len)
    u = T(rng.standard_normal(h.ndof))
    mat = mto.material()
    h.set_supports(h.side_dofs(0))
    h.build_elements(T(rho), mat)
    clean = h.indicator(u, T(rho), mat, maps=False)["eps_qr"].cpu().numpy()
    rho[e * d * d + d * d // 2] = bad
    got = h.indicator(u, T(rho), mat, maps=False)["eps_qr"].cpu().numpy()
    h.set_build_path(mto.BUILD_SIMT)
    want = h.indicator(u, T(rho), mat, maps=False)["eps_qr"].cpu().numpy()
    others = np.arange(nx * ny) != e
    np.testing.assert_array_equal(got[others], clean[others])
    assert np.isfinite(got[e]) == np.isfinite(want[e]) == bool(np.isfinite(bad))
    if np.isfinite(bad):
        assert abs(got[e] - want[e]) <= 1e-9 * abs(want[e])
    h.close()


@pytest.mark.parametrize("p,d", [(1, 8), (2, 4), (3, 8), (4, 3), (5, 8), (6, 2)])
@pytest.mark.parametrize("design", ["binary", "graded", "void"])
def test_qr_error_across_the_modulus_contrast(mto, p, d, design):
    """Elements that mix solid with 1e-9 void, or grade from one to the other: the QR error comes from the
    FP64 sums whatever the build path (equal bits), as the sliced rows keep only 2^-54 of the element's
    largest modulus; elements of moduli within a factor of 16 may take the rows (kappa of the pinned problem
    below 1e5 there, so 1e-9).  The maps of an adaptive step agree, and a sample agrees with the oracle to
    2^-50 of the pinned problem's condition number."""
    from oracle import indicators as oi
    from oracle import mesh as om
    from oracle.solve import K0_table
    nx, ny = 17, 9
    h = handle(mto, nx, ny, p, d)
    m = om.DPMesh(nx, ny, np.full(nx * ny, p), np.full(nx * ny, d))
    rng = np.random.default_rng(p + 10 * d)
    e = np.arange(nx * ny)
    c = (np.arange(d) + 0.5) / d
    x = (e % nx)[:, None, None] + c[None, None, :]
    y = (e // nx)[:, None, None] + c[None, :, None]
    s = np.sin(0.9 * x + 0.3 * y) + np.sin(0.4 * x - 1.1 * y) + 0.2
    rho = {"binary": (s > 0).astype(float), "graded": np.clip(1 / (1 + np.exp(-4 * s)), 1e-3, 1.0),
           "void": np.zeros_like(s)}[design].reshape(nx * ny, d * d)
    rho[5], rho[6] = 0.6, np.linspace(0.5, 0.9, d * d)
    u = rng.standard_normal(h.ndof)
    mat = mto.material()
    h.set_supports(h.side_dofs(0))
    h.build_elements(T(rho.ravel()), mat)
    got = h.indicator(T(u), T(rho.ravel()), mat)
    h.set_build_path(mto.BUILD_SIMT)
    ref = h.indicator(T(u), T(rho.ravel()), mat)
    a, b = got["eps_qr"].cpu().numpy(), ref["eps_qr"].cpu().numpy()
    E = 1e-9 + rho ** 3 * (1.0 - 1e-9)
    close = E.max(1) <= 15.9 * E.min(1)
    far = E.max(1) >= 16.1 * E.min(1)
    assert close.any() and (far.any() or design == "void")
    np.testing.assert_array_equal(a[far], b[far])
    assert np.abs(a - b)[close].max() <= 1e-9
    for k in ("p_new", "d_new", "theta"):
        np.testing.assert_array_equal(got[k].cpu().numpy(), ref[k].cpu().numpy())
    K0 = K0_table(p + 1, d, 0.3, 1.0, 1.0)
    fr = np.setdiff1d(np.arange(K0.shape[1]), oi.qr_fixed_local_dofs(p + 1))
    for k in np.concatenate([np.flatnonzero(far)[::7], [5, 6]]):
        kappa = np.linalg.cond(np.tensordot(E[k], K0, axes=(0, 0))[np.ix_(fr, fr)])
        want = oi.qr_error_element(p, d, rho[k], m.gather(k, u), 1.0, 1e-9, 0.3, 3.0)
        assert abs(a[k] - want) <= 2.0 ** -50 * kappa, (k, a[k], want, kappa)
    h.close()
