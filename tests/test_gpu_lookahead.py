"""The split path's look-ahead (few candidates, twelve block columns and more)
against the same candidates in a batch that factors without it: the same bits,
with candidates that fail in the first and in later block columns, in direct
calls, replayed plans and with either width of an update tile."""
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


# 12 to 15 block columns: pairs with and without a single column left over
@pytest.mark.parametrize("n,few,tile", [(1409, 1, 128), (1536, 7, 64), (1600, 48, 128), (1665, 20, 128), (1900, 5, 64)])
def test_lookahead_gives_the_batch_bits(gp, n, few, tile):
    ctx = gp.Context(0, update_tile=tile)
    g = np.random.default_rng(n)
    d, T, p, delta = 3, 70, 1.95, 1e-10
    x = dev(inputs.random_lhd(g, n, d))
    y = dev(inputs.y_sinsum(x.cpu().numpy()))
    # from far too smooth (not positive definite in split precision) to rough
    th = inputs.log_uniform_thetas(g, T, d, lo=-3.0, hi=2.0)
    th[0] = [1e-4, 1e-4, 1e-4]
    th[1:7] = np.geomspace(1e-2, 10.0, 6)[:, None]
    th = dev(th)
    whole = {k: v.cpu().numpy() for k, v in ctx.nll_batch(x, y, th, p, delta, "mixed").items()}
    failed = whole["status"] != 0
    assert failed.any() and not failed.all()
    part = th[:few].clone()
    plan = ctx.plan_nll_batch(x, y, part, p, delta, "mixed")
    for k in KEYS:
        plan.out[k].fill_(0)
    plan.launch()
    for out in [plan.out] + [ctx.nll_batch(x, y, part, p, delta, "mixed") for _ in range(4)]:
        for k in KEYS:
            assert np.array_equal(out[k].cpu().numpy(), whole[k][:few], equal_nan=True), k
    plan.free()


def test_timeout_under_lookahead_reports_and_recovers(gp):
    """A wait that nothing ends (the 5 ms hook) in the split GEMMs of a factor
    with look-ahead: the candidates it gives up come back GP_ETIMEOUT, the
    others with their bits, and the next call is normal."""
    ctx = gp.Context(0)
    g = np.random.default_rng(11)
    x = dev(inputs.random_lhd(g, 1500, 3))
    y = dev(inputs.y_sinsum(x.cpu().numpy()))
    th = dev(inputs.log_uniform_thetas(g, 8, 3, lo=0.0, hi=1.0))
    good = ctx.nll_batch(x, y, th, 1.95, 1e-6, "mixed")
    try:
        ctx.set_options(inject_timeout=1)
        bad = ctx.nll_batch(x, y, th, 1.95, 1e-6, "mixed")
        st = bad["status"].cpu().numpy()
    finally:
        ctx.set_options(inject_timeout=0)
    assert (st == -5).any() and np.isin(st, (0, -5)).all()
    assert np.isnan(bad["nll"].cpu().numpy()[st == -5]).all()
    assert np.array_equal(bad["nll"].cpu().numpy()[st == 0], good["nll"].cpu().numpy()[st == 0])
    again = ctx.nll_batch(x, y, th, 1.95, 1e-6, "mixed")
    for k in KEYS:
        assert np.array_equal(again[k].cpu().numpy(), good[k].cpu().numpy()), k
