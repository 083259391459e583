"""The field kernels on mirrored element pairs: kappa (FP64) and kappa32 (FP32)
against the oracle's dense exp(Phi xi) where the pairing has its edges: odd
meshes (the middle row or layer is its own partner), meshes of less than a
tile, one mode, odd numbers of modes, a truncated basis, and fields beyond the
normal range of exp.

Bound: with A the sum of |Phi_k xi_k| over the modes, an axis-by-axis sum of m
terms per axis with tables a few ulps off rounds to within dim (m + 6) + 8
units of A; kappa adds a few ulps of its own (FP32: 2^-21 for the hardware's
power of two)."""
import numpy as np
import pytest

from oracle import kle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def m():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2111_11788_gb300.build import build_library
    build_library()
    import paper_2111_11788_gb300.mlmc as mod
    mod.lib()
    return mod


def fields(m, dim, n, mpd, order, sigma2, xi):
    cfg = m.config(dim=dim, n_levels=1, coarse_cells=n, modes_per_dim=mpd, corr_len=0.2, sigma2=sigma2,
                   total_order=order)
    es, ne, count = m.elem_stride(dim, n), n ** dim, xi.shape[0]
    x = torch.from_numpy(np.ascontiguousarray(xi)).cuda()
    k64 = torch.full((count, es), -1.0, dtype=torch.float64, device="cuda")
    k32 = torch.full((count, es), -1.0, dtype=torch.float32, device="cuda")
    with m.Plan(cfg, torch.cuda.current_stream().cuda_stream) as plan:
        plan.kappa(0, x.data_ptr(), count, k64.data_ptr())
        plan.kappa32(0, x.data_ptr(), count, k32.data_ptr())
        torch.cuda.synchronize()
    return k64.cpu().numpy()[:, :ne], k32.cpu().numpy()[:, :ne].astype(np.float64)


@pytest.mark.parametrize("dim,n,mpd,order", [
    (2, 2, 1, -1), (2, 3, 2, -1), (2, 31, 3, -1), (2, 33, 8, -1), (2, 64, 5, 4), (2, 129, 1, -1), (2, 257, 32, 10),
    (3, 2, 1, -1), (3, 3, 3, -1), (3, 9, 4, 3), (3, 16, 7, -1), (3, 33, 2, -1), (3, 34, 16, 14),
])
def test_fields_against_oracle(m, dim, n, mpd, order):
    rng = np.random.default_rng(n * 31 + mpd)
    kept = None if order < 0 else order
    M = kle.n_modes(dim, mpd, kept)
    xi = rng.standard_normal((3, M))
    phi = kle.phi_matrix(dim, n, 0.2, 1.5, mpd, kept)
    ref, A = np.exp(xi @ phi.T), np.abs(xi) @ np.abs(phi).T
    k64, k32 = fields(m, dim, n, mpd, order, 1.5, xi)
    units = dim * (mpd + 6) + 8
    assert np.all(np.abs(k64 - ref) <= (units * A + 8) * 2.0 ** -53 * ref)
    assert np.all(np.abs(k32 - ref) <= ((units * A + 8) * 2.0 ** -24 + 2.0 ** -21) * ref)


def test_fields_beyond_the_range_of_exp(m):
    """One mode in 2D: x = xi Phi_0 up to +-1000; zero, subnormal, infinite and NaN results as exp gives them."""
    n = 16
    phi = kle.phi_matrix(2, n, 0.2, 1.0, 1)
    top = 1000.0 / phi.max()
    xi = np.array([[top], [-top], [0.7 * top], [-0.7 * top], [np.nan]])
    x = xi @ phi.T
    k64, _ = fields(m, 2, n, 1, -1, 1.0, xi)
    with np.errstate(over="ignore", under="ignore"):
        ref = np.exp(x)
    assert np.isnan(k64[4]).all()
    got, ref, x = k64[:4], ref[:4], x[:4]
    assert np.all(np.isinf(got[x > 710.5])) and np.all(got[x < -746.0] == 0.0)
    normal = np.abs(x) < 707.0
    assert normal.any() and np.all(np.abs(got - ref)[normal] <= 40 * 2.0 ** -53 * (1 + np.abs(x[normal])) * ref[normal])
