"""Device memory of a fermionic evaluator: its work buffers are those of n_max configurations until a
call takes local energies, and the results are the same bits before and after they grow."""
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


def test_buffers_are_those_of_n_max_until_energies_are_taken():
    # 6x6 D=4 chi=16 in float32: a configuration takes 1.6 MB of work buffers
    L1, L2, D, chi, n = 6, 6, 4, 16, 2
    th = binding.famp_init_theta(L1, L2, D, noise=0.1, seed=3)
    S = wl.fermion_support_configs(n, L1 * L2, 7)
    # every call once: kernels are loaded, and their local memory reserved, on first use
    warm = binding.FermionAmplitudes(L1, L2, D, chi, n, precision=binding.PEPS_TF32)
    warm.eval(th, S), warm.sweep(th, S, p=2, seed=1), warm.log_derivative(th, S)
    warm.local_energy(th, S, 1.0, 8.0, 4.0)
    warm.close()
    before = _free()
    f = binding.FermionAmplitudes(L1, L2, D, chi, n, precision=binding.PEPS_TF32)
    first = f.eval(th, S)
    swept = f.sweep(th, S, p=2, seed=1)
    rows = f.log_derivative(th, S)
    small = before - _free()
    assert small <= 64 * MB
    e1 = f.local_energy(th, S, 1.0, 8.0, 4.0)
    grown = before - _free()
    assert small < grown <= 4096 * MB
    e2 = f.local_energy(th, S, 1.0, 8.0, 4.0)
    assert before - _free() == grown
    for a, b in ((first, f.eval(th, S)), (swept, f.sweep(th, S, p=2, seed=1)), ([rows], [f.log_derivative(th, S)]),
                 (e1, e2)):
        assert all(np.array_equal(x, y) for x, y in zip(a, b))
    f.close()
    assert before - _free() <= 2 * MB


@pytest.mark.parametrize("prec", [binding.PEPS_FP64, binding.PEPS_TF32])
def test_energies_do_not_depend_on_the_evaluator(prec):
    # one configuration (4 hops a bond fill the buffers), some, more than eight per SM
    L1, L2, D, chi = 2, 3, 2, 4
    th = binding.famp_init_theta(L1, L2, D, noise=0.3, seed=5)
    S = wl.fermion_support_configs(1300, L1 * L2, 3)
    big = binding.FermionAmplitudes(L1, L2, D, chi, 1300, precision=prec)
    want = big.local_energy(th, S, 1.0, 8.0, 4.0)
    for n in (1, 40, 1300):
        f = binding.FermionAmplitudes(L1, L2, D, chi, n, precision=prec)
        for k in (0, 1300 - n):
            got = f.local_energy(th, S[k:k + n], 1.0, 8.0, 4.0)
            assert all(np.array_equal(a, b[k:k + n]) for a, b in zip(got, want))
        f.close()
    big.close()
