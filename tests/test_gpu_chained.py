"""Candidates evaluated a few at a time, where each launch is set up while the
one before it runs, against the same candidates in a batch whose launches are
plain: the same bits, in direct calls, under the gradient and in a replayed
plan."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1203_1269_gb300 import inputs

pytestmark = pytest.mark.gpu
KEYS = ("nll", "mu", "sigma2", "logdet", "status")


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1203_1269_gb300 import gp
    return gp.Context(0)


def dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


# (n, candidates of the plain batch): past 8 or 16 candidates or 128 (double)
# and 256 (split) candidates x block columns; at 1300 x 70 the substitutions
# have more than eight CTAs per SM and take their other variant
@pytest.mark.parametrize("prec,n,T", [("fp64", 40, 9), ("fp64", 256, 9), ("fp64", 257, 17), ("fp64", 700, 24),
                                      ("fp64", 1300, 12), ("mixed", 64, 257), ("mixed", 200, 130),
                                      ("mixed", 390, 65), ("mixed", 1300, 24), ("mixed", 1300, 70)])
def test_few_candidates_give_the_batch_bits(ctx, prec, n, T):
    g = np.random.default_rng(n + T)
    d, p, delta, few = 3, 1.95, 1e-6, 2
    x = dev(inputs.random_lhd(g, n, d))
    y = dev(inputs.y_sinsum(x.cpu().numpy()))
    th = dev(inputs.log_uniform_thetas(g, T, d, lo=-0.5, hi=1.0))
    whole = {k: v.cpu().numpy() for k, v in ctx.nll_batch(x, y, th, p, delta, prec).items()}
    part = th[:few].clone()
    plan = ctx.plan_nll_batch(x, y, part, p, delta, prec)
    for k in KEYS:
        plan.out[k].fill_(0)
    plan.launch()
    runs = [plan.out] + [ctx.nll_batch(x, y, part, p, delta, prec) for _ in range(5)]
    for out in runs:
        for k in KEYS:
            assert np.array_equal(out[k].cpu().numpy(), whole[k][:few], equal_nan=True), k
    plan.free()
    if prec == "fp64":
        out = ctx.nll_grad_batch(x, y, part, p, delta)
        assert np.array_equal(out["nll"].cpu().numpy(), whole["nll"][:few])
        again = ctx.nll_grad_batch(x, y, part, p, delta)
        assert np.array_equal(out["grad"].cpu().numpy(), again["grad"].cpu().numpy())
