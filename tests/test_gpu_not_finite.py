"""Parameters that are not finite, or overflow in float32: every engine returns from an evaluation and a
sweep, and the context then evaluates finite parameters to the bits of a fresh one."""
import numpy as np
import pytest

from paper_2409_05285_gb300 import binding
from paper_2409_05285_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2409_05285_gb300.build import build
    build()


@pytest.mark.parametrize("bad", [np.nan, np.inf, 1e30])
@pytest.mark.parametrize("prec,mode,launched", [
    (binding.PEPS_FP64, binding.PEPS_BLOCKS_NARROW, False), (binding.PEPS_FP64, binding.PEPS_BLOCKS_BATCHED, False),
    (binding.PEPS_FP64, binding.PEPS_BLOCKS_BATCHED, True), (binding.PEPS_FP32, binding.PEPS_BLOCKS_BATCHED, False),
    (binding.PEPS_TF32, binding.PEPS_BLOCKS_BATCHED, False), (binding.PEPS_TF32, binding.PEPS_BLOCKS_BATCHED, True)])
def test_evaluations_return(bad, prec, mode, launched):
    L1, L2, D, chi, n = 4, 5, 3, 7, 6
    th = wl.random_theta(L1, L2, D, seed=1, scale=0.3, diag_bias=1.0)
    S = wl.random_configs(L1, L2, n, seed=2)
    ref = binding.Context(L1, L2, D, chi, n, precision=prec, block_mode=mode)
    ref.set_theta(th)
    want = ref.eval_batch(S)
    ctx = binding.Context(L1, L2, D, chi, n, precision=prec, block_mode=mode)
    ctx.profile(launched)
    for part in (slice(None, None, 7), slice(0, 1), slice(None)):
        t = th.copy()
        t[part] = bad
        ctx.set_theta(t)
        ctx.set_configs(S)
        ctx.eval_batch(S)
        ctx.mc_sweep(1, p=2)
        assert ctx.get_configs().max() <= 3
    ctx.set_theta(th)
    assert all(np.array_equal(a, b) for a, b in zip(ctx.eval_batch(S), want))
    ctx.close()
    ref.close()
