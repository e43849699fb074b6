"""Phase timers of the double path: sweeps, row solves and trailing updates
each under their own phase, in the factor of up to two block columns and in the
larger one, with and without the look-ahead."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1203_1269_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,T", [(200, 3), (700, 2), (700, 17)])
def test_double_factor_fills_its_phases(n, T):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1203_1269_gb300 import gp
    ctx = gp.Context(0)
    g = np.random.default_rng(n + T)
    x = inputs.random_lhd(g, n, 3)
    args = [torch.as_tensor(np.ascontiguousarray(v), dtype=torch.float64, device="cuda")
            for v in (x, inputs.y_sinsum(x), inputs.log_uniform_thetas(g, T, 3, lo=0.0, hi=1.0))]
    ctx.set_timing(True)
    ctx.phase_times()
    before = ctx.launch_count()
    ctx.nll_batch(*args, 1.95, 1e-6, "fp64")
    phases = ctx.phase_times()
    assert sum(k for _, k in phases.values()) == ctx.launch_count() - before
    for name in ("assemble", "potrf", "trsm", "update", "solve"):
        ms, launches = phases[name]
        assert ms > 0 and launches > 0, name
