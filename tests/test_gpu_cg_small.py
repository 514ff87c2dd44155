"""The CG loop of small problems in one launch against the separate kernels
(peps_set_cg_product 2 and 3): the same bits in the update, the residual and the iteration count."""
import numpy as np
import pytest

from paper_2409_05285_gb300 import binding
from paper_2409_05285_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2409_05285_gb300.build import build
    build()


CASES = [  # (L1, L2, D, chi, precision, chains, exponent, tolerance)
    (4, 4, 2, 4, binding.PEPS_FP64, 2000, 2, 1e-10),
    (4, 4, 2, 4, binding.PEPS_TF32, 64, 1, 1e-10),    # 16-byte rows, float64 copy
    (3, 4, 3, 5, binding.PEPS_FP32, 131, 2, 1e-4),    # odd site slices, a chunk of three samples
    (4, 4, 3, 5, binding.PEPS_FP64, 7, 2, 1e-10),     # fewer samples than a block
    (2, 2, 1, 1, binding.PEPS_FP64, 1, 2, 1e-10),     # one sample, one entry a site
    (5, 5, 2, 4, binding.PEPS_FP32, 900, 1, 1e-2),
]


@pytest.mark.parametrize("case", CASES)
def test_small_cg_gives_the_bits_of_the_kernels(case):
    L1, L2, D, chi, prec, n, p, tol = case
    th = wl.random_theta(L1, L2, D, seed=n, scale=0.2, diag_bias=1.0)
    res = []
    # rows of whole 16-byte vectors in float32 take a float64 copy automatically (mode 3)
    vec = prec != binding.PEPS_FP64 and D % 2 == 0
    for mode in (0, 3 if vec else 2):
        ctx = binding.Context(L1, L2, D, chi, n, J2=0.2, precision=prec, seed=9)
        ctx.set_theta(th)
        ctx.set_cg_product(mode)
        out = []
        for _ in range(2):
            st = ctx.step(n_sweeps=1, p=p, tau=0.02, eps=1e-4, max_cg=60, cg_tol=tol)
            out += [ctx.get_theta(), st["cg_iters"], st["cg_resid"], st["E_site"]]
        res.append(out)
        ctx.close()
    assert all(np.array_equal(a, b) for a, b in zip(*res))
    assert np.all(np.isfinite(res[0][0]))
