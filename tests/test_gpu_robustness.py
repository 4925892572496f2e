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
