"""The split path's assembly with two candidates in a pair of FP32 lanes
against single candidates: the same bits, whatever the partner (none, refused,
or with entries that underflow), for every family, dimension and exponent
mode, and with more candidates than the theta of one group holds."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1203_1269_gb300 import inputs

pytestmark = pytest.mark.gpu
KEYS = ("nll", "mu", "sigma2", "logdet", "status")


def dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


@pytest.fixture(scope="module")
def gp():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1203_1269_gb300 import gp
    return gp


@pytest.mark.parametrize("corr,n,d,p,T", [("powexp", 1100, 1, 1.95, 33), ("powexp", 1100, 6, 1.0, 32),
                                          ("powexp", 1153, 10, 2.0, 35), ("powexp", 1100, 11, 1.5, 33),
                                          ("powexp", 1030, 10, 1.95, 1701), ("matern32", 1030, 16, 1.0, 1031),
                                          ("matern12", 130, 3, 1.0, 5), ("matern32", 129, 8, 1.0, 4),
                                          ("matern52", 300, 16, 1.0, 7)])
def test_pairs_give_the_single_candidate_bits(gp, corr, n, d, p, T):
    ctx = gp.Context(0, correlation=corr)
    g = np.random.default_rng(n + d)
    x = dev(inputs.random_lhd(g, n, d))
    y = dev(inputs.y_sinsum(x.cpu().numpy()))
    th = inputs.log_uniform_thetas(g, T, d, lo=0.0, hi=1.5)
    th[1] = -1.0                     # refused beside candidate 0
    th[3] = 1e30                     # every entry off the diagonal underflows
    whole = {k: v.cpu().numpy() for k, v in ctx.nll_batch(x, y, dev(th), p, 1e-6, "mixed").items()}
    assert (whole["status"][[0, 2]] == 0).all() and whole["status"][1] != 0
    for i in (0, 2, 3, T - 1):
        one = ctx.nll_batch(x, y, dev(th[i:i + 1]), p, 1e-6, "mixed")
        for k in KEYS:
            assert np.array_equal(one[k].cpu().numpy(), whole[k][i:i + 1], equal_nan=True), (i, k)
