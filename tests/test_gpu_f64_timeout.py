"""A bounded wait that runs out in the double path's tensor-core kernels (the
inject_timeout hook, 5 ms): in the factor's updates, with and without the
look-ahead, and in the gradient's inverse, whose kernels run after the
likelihood has been written.  The candidates given up come back GP_ETIMEOUT
with NaN outputs, the others with their bits, and the next call is normal."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1203_1269_gb300 import inputs

pytestmark = pytest.mark.gpu
ETIMEOUT = -5


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1203_1269_gb300 import gp
    return gp.Context(0)


def dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


def host(out):
    return {k: v.cpu().numpy() for k, v in out.items()}


# n = 200: the factor has no tensor-core kernel, so that the wait runs out in
# the inverse alone; 16 candidates are the most that look ahead
@pytest.mark.parametrize("call,n,T", [("nll", 700, 3), ("nll", 700, 17), ("grad", 200, 5), ("grad", 700, 3)])
def test_timeout_reports_and_recovers(ctx, call, n, T):
    g = np.random.default_rng(n + T)
    d, p, delta = 3, 1.95, 1e-6
    x = inputs.random_lhd(g, n, d)
    args = [dev(v) for v in (x, inputs.y_sinsum(x), inputs.log_uniform_thetas(g, T, d, lo=0.0, hi=1.0))]

    def run():
        return host(ctx.nll_grad_batch(*args, p, delta) if call == "grad" else ctx.nll_batch(*args, p, delta, "fp64"))

    good = run()
    try:
        ctx.set_options(inject_timeout=1)
        bad = run()
    finally:
        ctx.set_options(inject_timeout=0)
    again = run()
    assert np.all(good["status"] == 0)
    gone = bad["status"] == ETIMEOUT
    assert gone.any() and np.all(bad["status"][~gone] == 0)
    for k in good:
        if k != "status":
            assert np.isnan(bad[k][gone]).all(), k
            assert np.array_equal(bad[k][~gone], good[k][~gone]), k
        assert np.array_equal(again[k], good[k]), k
