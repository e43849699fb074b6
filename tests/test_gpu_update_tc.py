"""The double-precision factor (its products on the tensor cores from three
block columns on, in IEEE operations below) at ragged sizes, large nuggets, entries of L
next to 1, and failing pivots beyond the first block columns."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1203_1269_gb300 import inputs

pytestmark = pytest.mark.gpu
U = 2.0 ** -53


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1203_1269_gb300 import gp
    return gp.Context(0)


def dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


def unpack_lower(buf, n, nb=128):
    nt = (n + nb - 1) // nb
    full = np.zeros((nt * nb, nt * nb))
    idx = 0
    for J in range(nt):
        for I in range(J, nt):
            full[I * nb:(I + 1) * nb, J * nb:(J + 1) * nb] = buf[idx * nb * nb:(idx + 1) * nb * nb].reshape(nb, nb).T
            idx += 1
    return np.tril(full)[:n, :n]


def residual(ctx, x, th, p, delta):
    """max |R - L L'| against R as the library assembles it."""
    n = len(x)
    L, st = ctx.cholesky(dev(x), dev(th), p, delta, "fp64")
    assert st == 0
    L = unpack_lower(L.cpu().numpy(), n)
    R = unpack_lower(ctx.corr_assemble(dev(x), dev(th), p, delta, "tiles").cpu().numpy(), n)
    return np.max(np.abs(R - np.tril(L @ L.T)))


# Cholesky's backward error in doubles is at most (n + 1) u (1 + delta) entry
# by entry (rows of L have norm sqrt(1 + delta)), and the product L L' formed
# here for the check errs by n u (1 + delta) at most.
def bound(n, delta):
    return 2 * (n + 2) * U * (1.0 + delta)


@pytest.mark.parametrize("n", [1, 7, 31, 32, 33, 96, 127, 128, 129, 160, 225, 256, 257, 320, 383, 384, 385, 513, 700, 1025])
@pytest.mark.parametrize("d,lo", [(1, -1.0), (5, 0.0)])
def test_factor_residual(ctx, n, d, lo):
    g = np.random.default_rng(n + d)
    x = inputs.random_lhd(g, n, d)
    th = inputs.log_uniform_thetas(g, 1, d, lo=lo)[0]
    assert residual(ctx, x, th, 1.9, 1e-7) <= bound(n, 1e-7)


@pytest.mark.parametrize("delta", [1e-12, 1e-3, 1.0, 1e4])
def test_nuggets_and_near_duplicates(ctx, delta):
    """Points in close pairs, the second of each far down the order: entries of
    L off the diagonal next to 1 for small nuggets."""
    g = np.random.default_rng(12)
    x = inputs.random_lhd(g, 300, 3)
    x = np.concatenate([x, x + 1e-5])
    assert residual(ctx, x, np.array([3.0, 4.0, 5.0]), 1.0, delta) <= bound(600, delta)


@pytest.mark.parametrize("c", [256, 300, 511, 639])
def test_zero_pivot_beyond_the_first_columns(ctx, c):
    """Point c repeats point 3 and delta = 0: an exactly singular R whose
    factorisation fails at column c (or by rounding goes on with a pivot at
    rounding level); either way the other candidates are untouched."""
    from paper_1203_1269_gb300 import gp
    g = np.random.default_rng(c)
    x = inputs.random_lhd(g, 640, 3)
    y = inputs.y_sinsum(x)
    x[c] = x[3]
    th = np.array([[20.0, 30.0, 40.0], [25.0, 20.0, 30.0]])
    bad = ctx.nll_batch(dev(x), dev(y), dev(th), 1.0, 0.0, "fp64")
    assert all(int(s) in (0, gp.GP_ENOTPD) for s in bad["status"])
    # a batch with an invalid candidate in it: the others as alone
    mix = np.concatenate([th, [[-1.0, 1.0, 1.0]]])
    got = ctx.nll_batch(dev(x), dev(y), dev(mix), 1.0, 1e-6, "fp64")
    ref = ctx.nll_batch(dev(x), dev(y), dev(th), 1.0, 1e-6, "fp64")
    assert int(got["status"][2]) == gp.GP_EINVAL
    assert torch.equal(got["nll"][:2], ref["nll"]) and torch.equal(got["mu"][:2], ref["mu"])
