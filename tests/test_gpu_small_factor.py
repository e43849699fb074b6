"""The double factor of up to 256 points against the unblocked loops in IEEE
double on the host, bit for bit: pivots by sqrt, columns times the reciprocal,
every term one fma in the order of the columns (a second block column takes
the first one's terms as a sum of their own).  The kernel forms square root and
reciprocal from one float seed; pivots here run from 1e-8 to 1e3."""
import ctypes
import ctypes.util

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1203_1269_gb300 import inputs

pytestmark = pytest.mark.gpu

_libm = ctypes.CDLL(ctypes.util.find_library("m") or "libm.so.6")
_libm.fma.restype = ctypes.c_double
_libm.fma.argtypes = [ctypes.c_double] * 3
fma = np.vectorize(_libm.fma, otypes=[np.float64])
NB = 128


def tiles_of(v, n):
    nt = (n + NB - 1) // NB
    m = np.zeros((NB * nt, NB * nt))
    for (i, j), t in zip([(i, j) for j in range(nt) for i in range(j, nt)], v.cpu().numpy().reshape(-1, NB, NB)):
        m[NB * i:NB * i + NB, NB * j:NB * j + NB] = t.T
    return np.tril(m[:n, :n])


def unblocked(a):
    a = a.copy()
    n = len(a)
    for j0 in range(0, n, NB):
        j1 = min(j0 + NB, n)
        for c in range(j0, j1):
            a[c, c] = np.sqrt(a[c, c])
            a[c + 1:, c] *= 1.0 / a[c, c]
            for k in range(c + 1, j1):
                a[k:, k] = fma(-a[k:, c], a[k, c], a[k:, k])
        if j1 < n:
            acc = np.zeros((n - j1, n - j1))
            for c in range(j0, j1):
                acc = fma(a[j1:, c, None], a[None, j1:, c], acc)
            a[j1:, j1:] -= acc
    return np.tril(a)


@pytest.mark.parametrize("n,p,delta,reps", [(40, 1.95, 1e-8, 8), (40, 1.0, 0.0, 8), (33, 2.0, 1e-6, 8), (40, 1.5, 1e3, 8),
                                            (135, 1.95, 1e-8, 1)])
def test_ieee_bits(n, p, delta, reps):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1203_1269_gb300 import gp
    ctx = gp.Context(0)
    g = np.random.default_rng(n)
    for _ in range(reps):
        x = torch.as_tensor(np.ascontiguousarray(inputs.random_lhd(g, n, 2)), dtype=torch.float64, device="cuda")
        th = torch.as_tensor(inputs.log_uniform_thetas(g, 1, 2, lo=-0.5, hi=1.5)[0], dtype=torch.float64, device="cuda")
        nugget = delta * g.uniform(0.5, 1.0)
        factor, status = ctx.cholesky(x, th, p, nugget)
        r = tiles_of(ctx.corr_assemble(x, th, p, nugget, layout="tiles"), n)
        assert status == 0
        assert np.array_equal(tiles_of(factor, n), unblocked(r))
