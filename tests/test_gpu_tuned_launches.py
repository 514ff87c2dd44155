"""Launch shapes on the launched route (per-launch profiling selects it where a chain program would run):
grids, contraction chunks, chains per FFMA block and truncation blocks give the same bits; and lists
of chains longer than the grid of a contraction, against the same chains in small batches."""
import numpy as np
import pytest

from paper_2409_05285_gb300 import binding
from paper_2409_05285_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2409_05285_gb300.build import build
    build()


SHAPES = [  # (grid %, chains per FFMA block, contraction chunk, truncation threads)
    (50, 16, 16, 256), (200, 1, 32, 32), (100, 256, 8, 128), (400, 64, 64, 64), (1, 256, 8, 256)]
CASES = [  # (L1, L2, D, chi, precision, chains)
    (6, 6, 4, 16, binding.PEPS_TF32, 256),
    (6, 6, 4, 16, binding.PEPS_FP64, 64),
    (4, 5, 2, 3, binding.PEPS_FP32, 5),     # columns of a few elements, odd counts
    (5, 6, 3, 7, binding.PEPS_FP32, 3),     # 21 x 21: odd, tall and wide
    (4, 6, 4, 15, binding.PEPS_FP64, 300),  # several matrices per SM
    (4, 6, 5, 13, binding.PEPS_FP32, 2),    # 65 x 65: four lanes per pair
    (4, 6, 6, 20, binding.PEPS_FP64, 2),    # 120 x 120: long columns
]


@pytest.mark.parametrize("case", CASES)
@pytest.mark.parametrize("trunc64", [False, True])
def test_shapes_keep_the_bits(case, trunc64):
    L1, L2, D, chi, prec, n = case
    if trunc64 and prec == binding.PEPS_FP64:
        pytest.skip("float64 truncates in float64")
    ctx = binding.Context(L1, L2, D, chi, n, J2=0.2, precision=prec, seed=6)
    ctx.set_theta(wl.random_theta(L1, L2, D, seed=chi, scale=0.1, diag_bias=1.0))
    if trunc64:
        ctx.set_trunc_fp64(True)
    S = wl.random_configs(L1, L2, n, seed=3)
    want = ctx.eval_batch(S)
    ctx.profile(True)
    for grid, g, kc, tt in SHAPES:
        ctx.set_tune(grid, 12 * 1024, g, kc, 1, 96, tt)
        l0 = ctx.launches()
        got = ctx.eval_batch(S)
        assert ctx.launches() - l0 > 100
        assert all(np.array_equal(a, b) for a, b in zip(want, got)), (grid, g, kc, tt)
    ctx.close()


@pytest.mark.parametrize("prec", [binding.PEPS_TF32, binding.PEPS_FP32, binding.PEPS_FP64])
def test_lists_longer_than_the_grid(prec):
    L1, L2, D, chi, n, part = 4, 4, 4, 16, 6000, 500
    ctx = binding.Context(L1, L2, D, chi, n, J2=0.2, precision=prec, seed=6)
    ctx.set_theta(wl.random_theta(L1, L2, D, seed=chi, scale=0.1, diag_bias=1.0))
    S = wl.random_configs(L1, L2, n, seed=3)
    l0 = ctx.launches()
    whole = ctx.eval_batch(S)
    assert ctx.launches() - l0 > 100
    for k in range(0, n, part):
        l0 = ctx.launches()
        got = ctx.eval_batch(S[k:k + part])
        assert ctx.launches() - l0 < 10
        assert all(np.array_equal(a[k:k + part], b) for a, b in zip(whole, got)), k
    ctx.close()
