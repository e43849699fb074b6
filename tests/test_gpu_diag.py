"""The double-float diagonal block (k_diag_mixed) at the edges of its internal
blocks: 8-column steps, 16-row warp groups, 32-column lanes, 128-row tiles."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1203_1269_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1203_1269_gb300 import gp
    return gp.Context(0)


def dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


def first_tile(buf, n):
    """Rows and columns below min(n, 128) of tile (0, 0): column-major."""
    m = min(n, 128)
    return np.tril(buf.cpu().numpy()[:128 * 128].reshape(128, 128).T)[:m, :m]


@pytest.mark.parametrize("n", [1, 2, 7, 8, 9, 15, 16, 17, 31, 32, 33, 63, 64, 65, 96, 97, 120, 127, 128, 129])
def test_block_factor(ctx, n):
    """L of the first tile against LAPACK.  Double-float operations and the
    assembled entries are exact to 2^-44 or better, so |L - L_ref| is within
    (n + 2) cond(R) 2^-43 (both factors' backward errors)."""
    g = np.random.default_rng(900 + n)
    x = inputs.random_lhd(g, n, 3)
    th = np.array([20.0, 30.0, 40.0])
    L, st = ctx.cholesky(dev(x), dev(th), 1.0, 1e-3, "mixed")
    assert st == 0
    R = np.exp(-np.sum(th * np.abs(x[:, None, :] - x[None, :, :]), axis=2)) + 1e-3 * np.eye(n)
    ref = np.linalg.cholesky(R)[:128, :128]
    err = np.max(np.abs(first_tile(L, n) - ref))
    assert err <= (n + 2) * np.linalg.cond(R) * 2.0 ** -43


@pytest.mark.parametrize("delta", [1e29, 1e31])
def test_pivots_outside_the_float_seed_range(ctx, delta):
    """A nugget of 1e31 takes the pivots' double route, 1e29 the float seed's:
    L is sqrt(1 + delta) on the diagonal, R_ij / sqrt(1 + delta) below it."""
    g = np.random.default_rng(77)
    x = inputs.random_lhd(g, 40, 3)
    th = np.array([2.0, 3.0, 4.0])
    L, st = ctx.cholesky(dev(x), dev(th), 1.0, delta, "mixed")
    assert st == 0
    ref = np.exp(-np.sum(th * np.abs(x[:, None, :] - x[None, :, :]), axis=2)) / np.sqrt(delta)
    ref = np.tril(ref, -1) + np.sqrt(1.0 + delta) * np.eye(40)
    got = first_tile(L, 40)
    assert np.max(np.abs(got - ref) / ref.max()) <= 2.0 ** -43
    low = np.tril_indices(40, -1)
    assert np.max(np.abs(got[low] - ref[low])) <= 2.0 ** -43 * np.max(ref[low])


@pytest.mark.parametrize("c", [1, 7, 8, 15, 16, 31, 32, 64, 127])
def test_zero_pivot_is_reported(ctx, c):
    """Design point c repeats point 0 and delta = 0: the pivot of column c is
    exactly zero, in whichever of the block's steps it falls."""
    from paper_1203_1269_gb300 import gp
    g = np.random.default_rng(50 + c)
    x = inputs.random_lhd(g, 128, 3)
    x[c] = x[0]
    _, st = ctx.cholesky(dev(x), dev(np.array([20.0, 30.0, 40.0])), 1.0, 0.0, "mixed")
    assert st == gp.GP_ENOTPD
