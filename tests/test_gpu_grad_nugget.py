"""The gradient where the nugget dominates (R close to 11' + delta I): columns
of L^-1 are nearly constant over a block of rows there, so the leading digit
products of R^-1 = X'X come close to their largest value.  delta runs over a
factor of four, so that the columns' entries lie all over a binade."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
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


# Backward errors of n u in the factor and in R^-1 move the gradient by at most
# about n cond(R) u of its terms' size; both sides (the oracle's too) err so.
def tol(n, cond):
    return 4 * n * cond * 2.0 ** -53


@pytest.mark.parametrize("n,d,theta,p,delta", [
    (640, 2, 0.0, 1.95, 0.1), (640, 2, 1e-6, 1.95, 1e-2), (640, 3, 1e-5, 1.95, 1e-3),
    (1024, 6, 1e-6, 1.95, 1e-2), (1024, 6, 1e-5, 1.95, 2e-2), (1024, 2, 1e-4, 1.95, 0.1), (1024, 2, 1e-4, 1.95, 0.2),
    (1024, 2, 1e-4, 1.95, 0.4), (1024, 1, 1e-3, 2.0, 1.0), (1280, 2, 1e-2, 2.0, 1.0), (2048, 6, 1e-5, 1.95, 0.1)])
def test_nearly_constant_columns(ctx, n, d, theta, p, delta):
    g = np.random.default_rng(n + d)
    x = inputs.random_lhd(g, n, d)
    y = inputs.y_sinsum(x) + g.standard_normal(n)
    th = np.full((1, d), theta)
    got = ctx.nll_grad_batch(dev(x), dev(y), dev(th), p, delta)
    ref, _, st = oracle.nll_grad(x, y, th[0], p, delta)
    assert st == 0 and int(got["status"][0]) == 0
    gg = got["grad"][0].cpu().numpy()
    # R is 11' + delta I but for what theta takes off: cond(R) = n / delta + 1 at most
    assert np.max(np.abs(gg - ref)) <= tol(n, n / delta + 1) * np.max(np.abs(ref))
