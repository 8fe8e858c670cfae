"""Products that may start before their predecessor has finished (programmatic
dependent launch), in a chain that writes two buffers in turn: x -> y -> x ...,
each product reading what the one before it has just written into a buffer that
the one before that has read. On a stream and in a captured graph, from grids of
which many fit on the GPU at once to grids of several waves, the last two
vectors equal, bit for bit, those of the same products with the device
synchronised after each."""
import functools

import numpy as np
import pytest

from paper_2604_13433_gb300 import inputs as I

from _gpu import P, dev, need_gpu, torch

pytestmark = pytest.mark.gpu

KINDS = {  # encode options, pinned variant, vector type
    "fp16": (dict(fmt="fp16", D=15), 13, "float32"),
    "fp16_explicit": (dict(fmt="fp16", D=15, explicit_perm=True), 13, "float32"),
    "e8my": (dict(fmt="e8my", D=11), 13, "float32"),
    "fixed": (dict(fmt="fixed", D=15), 0, "float32"),
    "sell_f32": (dict(fmt="sell_f32"), 0, "float32"),
    "sell_f16": (dict(fmt="sell_f16"), 0, "float32"),
    "w16": (dict(fmt="w16_e4m3", D=7), 0, "float32"),
    "x16": (dict(fmt="fp16", D=15), 0, "float16"),
    "w64": (dict(fmt="w64_e11my", D=15), 0, "float64"),
}


@functools.lru_cache(maxsize=None)
def matrix(grid):
    """27-point pattern, values of both signs scaled so that products keep
    their size (spectral radius of independent entries: sqrt(27 var) = 1)."""
    csr = I.stencil27(grid, seed=1)
    g = np.random.default_rng(5)
    csr.val = (g.uniform(-1.0, 1.0, csr.nnz) / 3.0).astype(np.float32)
    return csr


@pytest.mark.parametrize("grid", [(8, 8, 8), (24, 24, 24), (61, 47, 53), (97, 96, 95)])
@pytest.mark.parametrize("kind", sorted(KINDS))
def test_chain_over_two_buffers(kind, grid):
    need_gpu()
    ps = P()
    opts, variant, dtype = KINDS[kind]
    steps = 16 if dtype == "float16" else 48  # (longer chains overflow binary16)
    csr = matrix(grid)
    A = ps.packsell_encode_csr(csr, **opts)
    if variant:
        ps.packsell_set_spmv_variant(A, variant)
    product = {"float32": ps.packsell_spmv, "float16": ps.packsell_spmv_x16,
               "float64": ps.packsell_spmv_f64}[dtype]
    start = dev(I.uniform(csr.n, seed=2, lo=-1.0, hi=1.0)).to(getattr(torch, dtype))
    a, b = start.clone(), torch.zeros_like(start)

    def chain(sync=False):
        u, v = a, b
        for _ in range(steps):
            product(A, u, v)
            if sync:
                torch.cuda.synchronize()
            u, v = v, u

    chain(sync=True)
    want = [a.clone(), b.clone()]
    assert torch.isfinite(want[0]).all() and want[0].abs().max() > 1e-4

    def check(what):
        torch.cuda.synchronize()
        assert torch.equal(a, want[0]) and torch.equal(b, want[1]), what

    for r in range(3):
        a.copy_(start)
        torch.cuda.synchronize()
        chain()
        check(f"stream, run {r}")
    a.copy_(start)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        chain()
    for r in range(3):
        a.copy_(start)
        torch.cuda.synchronize()
        graph.replay()
        check(f"graph, run {r}")
