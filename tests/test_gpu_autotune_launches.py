"""The tuner times what its shapes act on: launches, also where a call of the context's size would run
as a chain program, and leaves the choice between the two as it was."""
import numpy as np
import pytest

from paper_2409_05285_gb300 import binding

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2409_05285_gb300.build import build
    build()


@pytest.mark.parametrize("prec,D,chi,knobs", [(binding.PEPS_FP64, 2, 4, 4), (binding.PEPS_TF32, 4, 16, 7)])
def test_candidates_are_launched(prec, D, chi, knobs):
    # knobs: candidates besides the present values
    ctx = binding.Context(4, 4, D, chi, 64, J2=0.2, precision=prec, seed=4)
    ctx.mc_sweep(1, p=2)
    want = ctx.eval_batch(None)
    l0 = ctx.launches()
    ctx.eval_batch(None)
    assert ctx.launches() - l0 < 10
    ctx.profile(True)
    l0 = ctx.launches()
    ctx.eval_batch(None)
    one = ctx.launches() - l0
    ctx.profile(False)
    l0 = ctx.launches()
    ctx.autotune(reps=0)
    assert ctx.launches() == l0
    ctx.autotune(reps=2)
    # one evaluation to warm up and two each for the present shapes and every candidate
    assert ctx.launches() - l0 >= (3 + 2 * knobs) * one
    l0 = ctx.launches()
    assert all(np.array_equal(a, b) for a, b in zip(want, ctx.eval_batch(None)))
    assert ctx.launches() - l0 < 10
    ctx.close()
