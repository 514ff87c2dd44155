"""Chain programs of calls whose number of chains changes: one program for every count above sixteen
chains per SM, a bounded device memory for all of them, a route that does not depend on the
calls before, and the same bits whichever programs were dropped in between."""
import ctypes

import numpy as np
import pytest

from paper_2409_05285_gb300 import binding
from paper_2409_05285_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

MB = 1 << 20


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2409_05285_gb300.build import build
    build()


def _free():
    import torch
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


def test_many_counts_take_one_program():
    # a program of this evaluation takes 0.2 MB; device memory is handed out in pieces of 2 MB
    L1, L2, D, chi, n = 4, 4, 2, 4, 3000
    ctx = binding.Context(L1, L2, D, chi, n, J2=0.3, precision=binding.PEPS_FP64)
    ctx.set_theta(wl.random_theta(L1, L2, D, seed=1, scale=0.3, diag_bias=1.0))
    S = wl.random_configs(L1, L2, n, seed=2)
    want = ctx.eval_batch(S)
    before, l0 = _free(), ctx.launches()
    for k in range(64):
        m = n - 1 - 9 * k   # above 2432 = 16 x 152 chains
        assert all(np.array_equal(a[:m], b) for a, b in zip(want, ctx.eval_batch(S[:m])))
    assert ctx.launches() - l0 == 64
    assert before - _free() <= 4 * MB
    ctx.close()


def test_route_of_a_call_is_its_own():
    # 2.3e5 flops an operation: a program for 153 chains, launches for 300 (both two per SM)
    L1, L2, D, chi = 4, 4, 6, 36
    th = wl.random_theta(L1, L2, D, seed=1, scale=0.1, diag_bias=1.0)
    S = wl.random_configs(L1, L2, 300, seed=2)
    seen, out = [], []
    for order in ((153, 300), (300, 153)):
        ctx = binding.Context(L1, L2, D, chi, 300, J2=0.3, precision=binding.PEPS_TF32)
        ctx.set_theta(th)
        count, got = {}, {}
        for m in order:
            l0 = ctx.launches()
            got[m] = ctx.eval_batch(S[:m])
            count[m] = ctx.launches() - l0
        seen.append(count)
        out.append(got)
        ctx.close()
    assert seen[0] == seen[1]
    assert seen[0][153] < 10 < seen[0][300]
    assert all(np.array_equal(a, b) for m in (153, 300) for a, b in zip(out[0][m], out[1][m]))


@pytest.mark.parametrize("graphs", [False, True])
def test_dropped_programs_are_made_again(graphs):
    # 16 block shapes x 2 kinds of evaluation exceed the memory of the programs (256 KB a site)
    import torch
    L1, L2, D, chi, n = 4, 4, 2, 4, 2432
    side = torch.cuda.Stream()
    ctx = binding.Context(L1, L2, D, chi, n, J2=0.3, precision=binding.PEPS_FP64, seed=4,
                          stream=ctypes.c_void_p(side.cuda_stream))
    ctx.set_theta(wl.random_theta(L1, L2, D, seed=1, scale=0.3, diag_bias=1.0))
    ctx.set_graphs(graphs)
    S = wl.random_configs(L1, L2, n, seed=2)
    want = ctx.eval_batch(S)
    before = _free()
    for _ in range(2):
        for m in range(n, 0, -152):
            for with_O in (True, False):
                got = ctx.eval_batch(S[:m], with_O=with_O)
                assert all(np.array_equal(a[:m], b) for a, b in zip(want, got) if b is not None)
    if not graphs:   # captures take memory of their own
        assert before - _free() <= (4 * 4 * 256 * 1024) + 4 * MB
    ctx.close()


def test_fermionic_sweep_of_many_chains():
    # the proposals of a move apply to a number of chains of its own, thousands of them
    L1, L2, D, chi, n = 2, 3, 2, 4, 6000
    th = binding.famp_init_theta(L1, L2, D, noise=0.3, seed=3)
    S = wl.fermion_support_configs(n, L1 * L2, 7)
    out = []
    for prof in (False, True):
        f = binding.FermionAmplitudes(L1, L2, D, chi, n, precision=binding.PEPS_FP64)
        f.profile(prof)
        res = f.sweep(th, S, p=2, seed=1)
        before = _free()
        res = [*res, *f.sweep(th, res[0], p=2, seed=1, sweep0=1)]
        if not prof:
            assert before - _free() <= 2 * MB
        out.append(res)
        f.close()
    assert all(np.array_equal(a, b) for a, b in zip(*out))
