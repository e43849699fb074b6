"""Backward error R - L L' of the double factor, formed exactly enough (slices
of 20 bits, whose products are exact in double, added by TwoSum): the digits
that the products are cut into are rounded to nearest, so the error has no
preferred sign."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1203_1269_gb300 import inputs

pytestmark = pytest.mark.gpu


def dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


def lower(tiles, n):
    """The lower triangle held in the factorisation's tile layout."""
    nt = (n + 127) // 128
    m = torch.zeros(128 * nt, 128 * nt, dtype=torch.float64, device="cuda")
    pairs = [(i, j) for j in range(nt) for i in range(j, nt)]
    for (i, j), t in zip(pairs, tiles.reshape(-1, 128, 128)):
        m[128 * i:128 * i + 128, 128 * j:128 * j + 128] = t.T
    return torch.tril(m[:n, :n])


def residual(r, low):
    """R - L L' (lower triangle) to about 1e-26."""
    parts, rest = [], low
    for i in range(4):
        unit = 2.0 ** (-20 * (i + 1))
        parts.append(torch.round(rest / unit) * unit)
        rest = rest - parts[-1]
    hi, err = r.clone(), torch.zeros_like(r)
    for i, j in sorted(((i, j) for i in range(4) for j in range(4)), key=sum):
        b = -(parts[i] @ parts[j].T)
        s = hi + b
        bb = s - hi
        err += (hi - (s - bb)) + (b - bb)
        hi = s
    return torch.tril(hi + err)


@pytest.mark.parametrize("n,d,p,delta", [(1000, 6, 1.5, 1e-6), (2000, 10, 1.5, 1e-7), (2100, 12, 1.9, 1e-6)])
def test_error_of_the_factor_has_no_sign(n, d, p, delta):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1203_1269_gb300 import gp
    ctx = gp.Context(0)
    g = np.random.default_rng(n + d)
    x = dev(inputs.random_lhd(g, n, d))
    th = dev(inputs.log_uniform_thetas(g, 1, d, lo=-1.0)[0])
    factor, status = ctx.cholesky(x, th, p, delta)
    assert status == 0
    e = residual(lower(ctx.corr_assemble(x, th, p, delta, layout="tiles"), n), lower(factor, n))
    count = n * (n + 1) / 2
    mean, rms = float(e.sum()) / count, float((e ** 2).sum() / count) ** 0.5
    # errors of one sign have a mean about as large as their root mean square;
    # of independent ones it is the 1/sqrt(n) of a row's common part, and ties
    # (rounded away from zero, in one binade of the entries) add a little
    assert abs(mean) <= rms / 4
    # IEEE multiply-adds: half an ulp of an entry below 1 + delta per panel
    assert float(e.abs().max()) <= (n // 128 + 1) * 2.0 ** -53
