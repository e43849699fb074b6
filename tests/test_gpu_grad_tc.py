"""The gradient with R^-1 formed on the tensor cores: ragged sizes around the
tile and half-tile edges, columns of L^-1 of very different sizes, and the
same bits alone and in a batch."""
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


@pytest.mark.parametrize("n", [1, 2, 63, 64, 65, 127, 128, 129, 192, 257, 384, 385])
def test_gradient_sizes(ctx, n):
    g = np.random.default_rng(4000 + n)
    x = inputs.random_lhd(g, n, 3)
    y = inputs.y_trig2(x) + x[:, 2]
    th = inputs.log_uniform_thetas(g, 2, 3, lo=0.3, hi=1.0)
    got = ctx.nll_grad_batch(dev(x), dev(y), dev(th), 1.8, 1e-4)
    for t in range(2):
        ref, _, st = oracle.nll_grad(x, y, th[t], 1.8, 1e-4)
        if st != 0:
            assert int(got["status"][t]) == st
            continue
        R = oracle.corr_matrix(x, th[t], 1.8, 1e-4)
        gg = got["grad"][t].cpu().numpy()
        assert np.max(np.abs(gg - ref)) <= tol(n, np.linalg.cond(R)) * max(1.0, np.max(np.abs(ref)))


def test_columns_of_very_different_sizes(ctx):
    """Pairs of points 1e-6 apart next to isolated ones: columns of L^-1 from
    about 1 to about 1e3 in the same tiles."""
    g = np.random.default_rng(99)
    x = inputs.random_lhd(g, 200, 4)
    x = np.concatenate([x, x[:60] + 1e-6])
    x = x[g.permutation(len(x))]
    y = inputs.y_sinsum(x)
    th = np.array([[8.0, 9.0, 10.0, 7.0]])
    got = ctx.nll_grad_batch(dev(x), dev(y), dev(th), 1.0, 1e-8)
    ref, _, st = oracle.nll_grad(x, y, th[0], 1.0, 1e-8)
    assert st == 0 and int(got["status"][0]) == 0
    cond = np.linalg.cond(oracle.corr_matrix(x, th[0], 1.0, 1e-8))
    gg = got["grad"][0].cpu().numpy()
    assert np.max(np.abs(gg - ref)) <= tol(len(x), cond) * np.max(np.abs(ref))


@pytest.mark.parametrize("n", [200, 300, 700, 2000])
def test_alone_and_in_a_batch(ctx, n):
    g = np.random.default_rng(n)
    x = inputs.random_lhd(g, n, 5)
    y = inputs.y_sinsum(x)
    th = inputs.log_uniform_thetas(g, 20, 5, lo=-0.5, hi=1.0)
    th[3] = -1.0                                   # one invalid candidate among them
    big = ctx.nll_grad_batch(dev(x), dev(y), dev(th), 1.9, 1e-6)
    for t in (0, 4, 19):
        one = ctx.nll_grad_batch(dev(x), dev(y), dev(th[t:t + 1]), 1.9, 1e-6)
        assert torch.equal(one["grad"][0], big["grad"][t]) and torch.equal(one["nll"][0], big["nll"][t])
    assert torch.isnan(big["grad"][3]).all()
