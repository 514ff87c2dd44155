"""The shared-memory truncation kernel (one-sided Jacobi with cached column norms) at the shapes
that select its variants: odd column counts, wide bonds with accumulated right vectors, columns
of one to many 16-byte vectors per lane, columns too long for registers, few and many matrices
per SM, several block sizes."""
import numpy as np
import pytest

from paper_2409_05285_gb300 import binding
from paper_2409_05285_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2409_05285_gb300.build import build
    build()


SHAPES = [  # (L1, L2, D, chi, n)
    (4, 5, 2, 3, 5),       # columns of a few elements, odd counts
    (5, 6, 3, 7, 3),       # 21 x 21: odd, tall and wide
    (4, 6, 4, 15, 300),    # 60 x 60, several matrices per SM
    (4, 6, 5, 13, 2),      # 65 x 65: four lanes per pair
    (4, 6, 6, 20, 2),      # 120 x 120: long columns (float64: read twice)
]


@pytest.mark.parametrize("shape", SHAPES)
def test_truncation_variants(shape):
    # Float64: the batched engine (this kernel) against the per-block engine, which runs the
    # general Jacobi routine, at the parity bounds (1e-10 in log|rho|, 1e-9 in the energies).
    # Float32: the same bits for every block size, and within the FP32 tolerance (2e-4) of
    # float64 on these near-product states.
    L1, L2, D, chi, n = shape
    th = wl.random_theta(L1, L2, D, seed=D * 100 + chi, scale=0.1, diag_bias=1.0)
    S = 3 * np.random.default_rng(chi).integers(0, 2, (n, L1 * L2)).astype(np.uint8)
    res = {}
    for name, prec, mode in (("narrow", binding.PEPS_FP64, binding.PEPS_BLOCKS_NARROW),
                             ("batched", binding.PEPS_FP64, binding.PEPS_BLOCKS_BATCHED),
                             ("fp32", binding.PEPS_FP32, binding.PEPS_BLOCKS_BATCHED),
                             ("trunc64", binding.PEPS_FP32, binding.PEPS_BLOCKS_BATCHED)):
        k = n if prec != binding.PEPS_FP64 else min(n, 8)
        ctx = binding.Context(L1, L2, D, chi, k, precision=prec, block_mode=mode)
        ctx.set_theta(th)
        if name == "trunc64":
            ctx.set_trunc_fp64(True)
        res[name] = ctx.eval_batch(S[:k], with_O=False)[:4]
        if name in ("fp32", "trunc64"):
            t = ctx.autotune(reps=0)
            for tt in (32, 128, 256):
                ctx.set_tune(t["grid_pct"], t["db_bytes"], t["ffma_g"], t["kc_max"], t["pipelined"],
                             t["stage_kb"], tt)
                again = ctx.eval_batch(S[:k], with_O=False)[:4]
                assert all(np.array_equal(a, b) for a, b in zip(res[name], again)), (name, tt)
        ctx.close()
    la, sg, es, ea = res["narrow"]
    k, scale = len(la), max(1.0, float(np.max(np.abs(res["narrow"][2]))))
    for name, tl, te in (("batched", 1e-10, 1e-9), ("fp32", 2e-4, 2e-4), ("trunc64", 2e-4, 2e-4)):
        b = [x[:k] for x in res[name]]
        assert np.array_equal(b[1], sg), name
        assert np.max(np.abs(b[0] - la)) <= tl, (name, np.max(np.abs(b[0] - la)))
        assert max(np.max(np.abs(b[2] - es)), np.max(np.abs(b[3] - ea))) <= te * scale, name
