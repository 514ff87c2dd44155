"""Proposals that change nothing are left out: evaluations of batches in which no chain, every
chain or some chains take an exchange on each bond, on both routes, against the oracle."""
import numpy as np
import pytest

from oracle import peps
from oracle.lattice import Lattice
from paper_2409_05285_gb300 import binding
from paper_2409_05285_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


def _batch(kind, n, L1, L2):
    stagger = (np.add.outer(np.arange(L1), np.arange(L2)) % 2).reshape(-1)
    if kind == "aligned":      # no exchange of neighbours changes anything
        return np.full((n, L1 * L2), 3, np.uint8)
    S = np.repeat((3 * stagger)[None].astype(np.uint8), n, 0)   # every one does
    if kind == "mixed":
        S[1::3] = 0
        S[2::3] = np.random.default_rng(n).integers(0, 4, S[2::3].shape)
    return S


@pytest.mark.parametrize("n", [1, 33, 130])
@pytest.mark.parametrize("kind", ["aligned", "staggered", "mixed"])
@pytest.mark.parametrize("prec,D,chi", [(binding.PEPS_FP64, 2, 4), (binding.PEPS_TF32, 4, 16)])
def test_exchanges_of_some_chains(kind, n, prec, D, chi):
    L1, L2, J2 = 3, 4, 0.4
    lat = Lattice(L1, L2, D, J1=1.0, J2=J2)
    th = wl.random_theta(L1, L2, D, seed=2, scale=0.1, diag_bias=1.0)
    S = _batch(kind, n, L1, L2)
    out = []
    for prof in (False, True):
        ctx = binding.Context(L1, L2, D, chi, n, J2=J2, precision=prec, seed=5)
        ctx.set_theta(th)
        ctx.profile(prof)
        ev = ctx.eval_batch(S, with_O=True)
        ctx.set_configs(S)
        ctx.mc_sweep(1, p=2)
        out.append([*ev, ctx.get_configs()])
        ctx.close()
    assert all(np.array_equal(a, b) for a, b in zip(*out))
    # float64: rounding of sums of order one; TF32: the mixed path's bound on resolved states
    tol = 1e-9 if prec == binding.PEPS_FP64 else 5e-2
    for k in range(min(n, 3)):
        r = peps.eval_sample(lat, th, S[k], chi)
        for got, want in ((out[0][0][k], r["log_abs"]), (out[0][2][k], r["e_sys"]), (out[0][3][k], r["e_anc"])):
            assert abs(got - want) < tol * max(1.0, abs(want))
