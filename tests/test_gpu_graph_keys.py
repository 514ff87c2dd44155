"""Captured launch sequences (peps_set_graphs) of evaluations that share buffers with an earlier one
but not its number of configurations or its other arrays: the bits of direct launches, on the
sizes that run as a chain program and on those that are launched operation by operation."""
import ctypes

import numpy as np
import pytest

from paper_2409_05285_gb300 import binding
from paper_2409_05285_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

SHAPES = [  # (L1, L2, D, chi, precision, larger and smaller batch)
    (4, 4, 2, 4, binding.PEPS_FP64, 100, 60),     # program
    (4, 4, 4, 16, binding.PEPS_TF32, 100, 60),    # program on the tensor cores
    (4, 4, 6, 36, binding.PEPS_TF32, 260, 220),   # launched (float operations above the program's)
]


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2409_05285_gb300.build import build
    build()


def _context(shape, graphs):
    import torch
    L1, L2, D, chi, prec, big, _ = shape
    side = torch.cuda.Stream()   # stream capture needs a stream other than the legacy default
    ctx = binding.Context(L1, L2, D, chi, big, J2=0.3, precision=prec, seed=3,
                          stream=ctypes.c_void_p(side.cuda_stream))
    ctx.set_theta(wl.random_theta(L1, L2, D, seed=chi, scale=0.1, diag_bias=1.0))
    ctx.set_graphs(graphs)
    return ctx, side


def _batch(shape, n, seed):
    return wl.random_configs(shape[0], shape[1], n, seed=seed)


@pytest.mark.parametrize("shape", SHAPES)
def test_host_batches_of_changing_size(shape):
    big, small = shape[5], shape[6]
    out = []
    for graphs in (False, True):
        ctx, _ = _context(shape, graphs)
        got = []
        for k, (n, with_O) in enumerate(((big, True), (small, False), (big, False), (small, True), (big, True))):
            got += [x for x in ctx.eval_batch(_batch(shape, n, k), with_O=with_O) if x is not None]
        assert (ctx.graphs_captured() > 0) == graphs
        out.append(got)
        ctx.close()
    assert len(out[0]) == len(out[1])
    assert all(np.array_equal(a, b) for a, b in zip(*out))


@pytest.mark.parametrize("shape", SHAPES)
def test_device_batches_into_other_arrays(shape):
    import torch
    big, small = shape[5], shape[6]
    out = []
    for graphs in (False, True):
        ctx, side = _context(shape, graphs)
        odt = torch.float64 if shape[4] == binding.PEPS_FP64 else torch.float32
        S = torch.empty((big, shape[0] * shape[1]), dtype=torch.uint8, device="cuda")
        O = torch.empty((big, ctx.No), dtype=odt, device="cuda")
        arrays = [[torch.empty(big, dtype=d, device="cuda")
                   for d in (torch.float64, torch.int8, torch.float64, torch.float64)] for _ in range(2)]
        got = []
        for k, (n, a, with_O) in enumerate(((big, 0, True), (big, 1, True), (small, 0, True), (big, 0, False),
                                            (small, 1, False), (big, 1, True))):
            S[:n] = torch.from_numpy(_batch(shape, n, k)).cuda()
            for t in (*arrays[0], *arrays[1], O):
                t.fill_(7)
            torch.cuda.synchronize()
            ctx.eval_batch_device(S[:n], *arrays[a], O if with_O else None)
            got += [t.cpu().numpy() for t in (*arrays[0], *arrays[1], O)]
        assert (ctx.graphs_captured() > 0) == graphs
        out.append(got)
        ctx.close()
    assert all(np.array_equal(a, b) for a, b in zip(*out))


def test_graphs_of_many_arrays_stay_bounded():
    shape = SHAPES[0]
    ctx, _ = _context(shape, True)
    ref, _ = _context(shape, False)
    for n in range(1, 81):
        S = _batch(shape, n, n)
        assert all(np.array_equal(a, b) for a, b in zip(ctx.eval_batch(S), ref.eval_batch(S)))
        assert ctx.graphs_captured() <= 64
    ctx.close()
    ref.close()
