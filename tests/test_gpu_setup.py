"""Shared-memory limits are set by the launches that need them: contexts of several threads, made and
freed at the same time, launch kernels of more than 48 KB of shared memory on both routes."""
import threading

import numpy as np
import pytest

from paper_2409_05285_gb300 import binding
from paper_2409_05285_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2409_05285_gb300.build import build
    build()


def _evaluate(prec, launched, out, k):
    L1, L2, D, chi, n = 4, 4, 4, 16, 8
    ctx = binding.Context(L1, L2, D, chi, n, precision=prec, seed=1)
    ctx.set_theta(wl.random_theta(L1, L2, D, seed=2, scale=0.1, diag_bias=1.0))
    ctx.profile(launched)
    out[k] = ctx.eval_batch(wl.random_configs(L1, L2, n, seed=3))
    ctx.close()


@pytest.mark.parametrize("prec", [binding.PEPS_FP64, binding.PEPS_FP32, binding.PEPS_TF32])
def test_contexts_of_several_threads(prec):
    out = [None] * 8
    threads = [threading.Thread(target=_evaluate, args=(prec, k % 2 == 1, out, k)) for k in range(8)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for o in out:
        assert o is not None and all(np.array_equal(a, b) for a, b in zip(o, out[0]))
