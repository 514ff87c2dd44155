"""Chain programs (one launch per evaluation, sweep or draw) against the launches per operation,
which profiling selects: the same bits on the same context, over bond dimensions, precisions and
chain counts that choose other block shapes and operation forms."""
import numpy as np
import pytest

from paper_2409_05285_gb300 import binding
from paper_2409_05285_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2409_05285_gb300.build import build
    build()


CASES = [  # (L1, L2, D, chi, J2, precision, chains)
    (3, 4, 3, 5, 0.4, binding.PEPS_FP64, 40),     # odd bonds, Householder rows not of four
    (2, 2, 1, 1, 0.0, binding.PEPS_FP64, 3),      # bonds of one
    (4, 4, 2, 4, 0.0, binding.PEPS_FP64, 3000),   # one warp per chain
    (5, 4, 2, 3, 0.3, binding.PEPS_TF32, 1700),   # no tensor-core contraction
    (4, 3, 4, 9, 0.3, binding.PEPS_FP32, 33),     # split tensor-core products
    (4, 4, 4, 12, 0.3, binding.PEPS_TF32, 1),     # Gram factors, one chain
    (5, 4, 4, 16, 0.0, binding.PEPS_TF32, 310),   # three chains per SM
    (4, 4, 6, 20, 0.2, binding.PEPS_TF32, 20),    # rows and columns past one tile, long columns
    (3, 3, 5, 11, 0.1, binding.PEPS_FP32, 9),     # element-wise operand gathers
]


@pytest.mark.parametrize("case", CASES)
def test_program_gives_the_bits_of_the_launches(case):
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
        S1 = ctx.get_configs()
        ev = ctx.eval_batch(None, with_O=True)               # with the sweep's up environments
        ev2 = ctx.eval_batch(S1[::-1].copy(), with_O=True)   # a caller's configurations
        ctx.mc_sweep(2, p=2)
        out.append([S1, ctx.get_configs(), *ev, *ev2])
        ctx.close()
    assert launches[0] < 10 < launches[1]
    assert all(np.array_equal(a, b) for a, b in zip(*out))


@pytest.mark.parametrize("prec", [binding.PEPS_FP64, binding.PEPS_TF32])
def test_direct_draws_on_both_routes(prec):
    L1, L2, D, chi, n = 4, 4, 2, 8, 50
    th = wl.random_theta(L1, L2, D, seed=4, scale=0.3, diag_bias=1.0)
    u = np.random.default_rng(1).random((n, L1 * L2))
    res = []
    for prof in (False, True):
        ctx = binding.Context(L1, L2, D, chi, n, precision=prec)
        ctx.set_theta(th)
        ctx.profile(prof)
        res.append((ctx.direct_draw(u, b_d=0.9), ctx.get_configs()))
        ctx.close()
    assert np.array_equal(res[0][0], res[1][0]) and np.array_equal(res[0][1], res[1][1])


@pytest.mark.parametrize("prec", [binding.PEPS_FP64, binding.PEPS_TF32])
def test_fermionic_calls_on_both_routes(prec):
    L1, L2, D, chi, n = 3, 4, 4, 9, 20
    th = binding.famp_init_theta(L1, L2, D, noise=0.1, seed=3)
    S = wl.fermion_support_configs(n, L1 * L2, 7)
    res = []
    for prof in (False, True):
        f = binding.FermionAmplitudes(L1, L2, D, chi, n, precision=prec)
        f.profile(prof)
        res.append([*f.eval(th, S), *f.local_energy(th, S, 1.0, 8.0, 4.0), f.log_derivative(th, S),
                    *f.sweep(th, S, p=2, seed=1)])
        f.close()
    assert all(np.array_equal(a, b) for a, b in zip(*res))
