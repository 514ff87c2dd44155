"""Launched kernels against the chain program's forms of the same operations, the same bits: Gram
factors in panels (rows 75, 80 and 216: remainders of 16, none, a matrix per SM), dot products of
long vectors by blocks, operands contiguous in pairs (bonds of 6), split and not."""
import numpy as np
import pytest

from paper_2409_05285_gb300 import binding
from paper_2409_05285_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

CASES = [  # (L1, L2, D, chi, J2, precision, chains)
    (4, 4, 6, 36, 0.2, binding.PEPS_TF32, 5),
    (4, 4, 5, 15, 0.3, binding.PEPS_TF32, 7),
    (4, 5, 4, 20, 0.0, binding.PEPS_TF32, 33),
    (4, 3, 6, 12, 0.2, binding.PEPS_FP32, 9),
]


@pytest.mark.parametrize("case", CASES)
def test_launched_forms_give_the_programs_bits(case):
    L1, L2, D, chi, J2, prec, n = case
    th = wl.random_theta(L1, L2, D, seed=chi, scale=0.1, diag_bias=1.0)
    out, launches = [], []
    for prof in (False, True):
        ctx = binding.Context(L1, L2, D, chi, n, J2=J2, precision=prec, seed=5)
        ctx.set_theta(th)
        ctx.profile(prof)
        l0 = ctx.launches()
        ctx.mc_sweep(1, p=1)
        launches.append(ctx.launches() - l0)
        out.append([ctx.get_configs(), *ctx.eval_batch(None, with_O=True)])
        ctx.close()
    assert launches[0] < 10 < launches[1]
    assert all(np.array_equal(a, b) for a, b in zip(*out))
