"""The encoder at the edges of its kernels' tiles, against the oracle's encoder
byte for byte: runs of 128 nonzeros per warp of 32 rows, rounds of 16 entries
per row, rows of 65,536 words and more in the sigma sort, CSR order, and the
memory that the library keeps between calls."""
import numpy as np
import pytest

import oracle as O
from paper_2604_13433_gb300 import inputs as I

from _gpu import FMT, P, assert_same_encoding, dev, need_gpu, torch

pytestmark = pytest.mark.gpu

EDGES = [0, 1, 15, 16, 17, 31, 32, 33, 127, 128, 129, 0, 0, 300] * 5 + [2] * 70 + [0, 5]


def _matrix(lengths, m, seed):
    rng = np.random.default_rng(seed)
    rowptr = np.concatenate([[0], np.cumsum(lengths)]).astype(np.int64)
    col = np.concatenate([np.sort(rng.choice(m, size=k, replace=False)) for k in lengths])
    return I.CSR(n=len(lengths), m=m, rowptr=rowptr, col=col.astype(np.int32),
                 val=rng.standard_normal(rowptr[-1]).astype(np.float32))


@pytest.mark.parametrize("f64", [False, True])
@pytest.mark.parametrize("fmt,D", [("fp16", 15), ("e8my", 3), ("e8my", 11)])
@pytest.mark.parametrize("C,sigma,lengths,m", [
    (32, 256, EDGES, 40000), (32, 1, EDGES, 40000), (1, 1, EDGES, 40000), (1, 64, EDGES, 40000),
    (8, 48, EDGES, 3000), (32, 64, [7], 50), (1, 1, [7], 50),
    (32, 256, [3, 66000, 65535, 65536, 0, 66000] + [4] * 40, 70000)])
def test_encode_edges(f64, fmt, D, C, sigma, lengths, m):
    need_gpu()
    csr = _matrix(lengths, m, seed=len(lengths) + D)
    if f64:
        csr.val = csr.val.astype(np.float64) * (1 + 2.0 ** -30)
    A = P().packsell_encode_csr(csr, fmt=fmt, D=D, C=C, sigma=sigma)
    assert_same_encoding(A, O.encode(csr, C=C, sigma=sigma, D=D, fmt=FMT[fmt]))


@pytest.mark.parametrize("C", [1, 32])
def test_encode_refuses_values_after_the_structure(C):
    """A value that the format cannot hold is found while the words are
    scattered; the call still refuses, and names the value."""
    need_gpu()
    ps = P()
    csr = _matrix([20] * 100, 500, seed=1)
    csr.val[1234] = np.inf
    with pytest.raises(ps.PackSELLError) as e:
        ps.packsell_encode_csr(csr, C=C, sigma=1)
    assert e.value.code == 3 and "1234" in str(e.value)


def test_encode_on_streams_reuses_memory():
    """Matrices made and dropped on two streams in turn (their memory goes back
    to the library's pool and is used again) give the words of a first one."""
    need_gpu()
    ps = P()
    csr = I.stencil27((20, 19, 18), seed=3)
    enc = O.encode(csr, C=32, sigma=256, D=15, fmt=FMT["fp16"])
    rp, cl, vl = dev(csr.rowptr), dev(csr.col), dev(csr.val)
    x = dev(I.uniform(csr.m, seed=4))
    want = None
    streams = [torch.cuda.Stream() for _ in range(2)]
    for k in range(8):
        s = streams[k % 2]
        s.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(s):
            A = ps.packsell_encode(rp, cl, vl, csr.n, csr.m)
            y = ps.packsell_spmv(A, x)
        s.synchronize()
        want = y if want is None else want
        assert torch.equal(y, want)
        if k >= 6:
            assert_same_encoding(A, enc)
        del A


@pytest.mark.parametrize("n", [1, 255, 4095, 4096, 4097, 9000])
@pytest.mark.parametrize("kind", ["short", "zipf", "near", "empty"])
def test_csr_order_items_cover_the_rows(n, kind):
    """CSR-order products over matrices whose items are cut at the edges of the
    device cut's chunks and tiles (rows at the tile limits of the three kernels,
    long rows, runs of empty rows): variant 11 gives the bits of the
    thread-per-row kernel, variant 14 and the SpMM stay within gamma_w, and a
    batch of the matrix gives variant 14's bits."""
    need_gpu()
    ps = P()
    rng = np.random.default_rng(n)
    lengths = {"short": rng.integers(0, 3, n), "zipf": np.minimum(rng.zipf(2.0, n), 900),
               "near": rng.choice([1, 124, 125, 126, 252, 253, 254, 256, 257], n, p=[0.92] + [0.01] * 8),
               "empty": np.where(rng.random(n) < 0.999, 0, 700)}[kind]
    csr = _matrix([int(v) for v in lengths], 1000, seed=n + 1)
    A = ps.packsell_encode_csr(csr, C=1, sigma=1)
    deq = O.encode(csr, C=1, sigma=1, D=15, fmt=FMT["fp16"]).deq
    x = I.uniform(csr.m, seed=2)
    y = {}
    for v in (1, 11, 14):
        ps.packsell_set_spmv_variant(A, v)
        y[v] = ps.packsell_spmv(A, dev(x))
    assert torch.equal(y[1], y[11])
    ref = O.csr_spmv_f64(csr, deq, x.astype(np.float64))
    u = 2.0 ** -24
    w = 2.0 * csr.row_lengths() + 1
    tol = w * u / (1 - w * u) * O.csr_spmv_f64(csr, np.abs(deq), np.abs(x).astype(np.float64))
    assert np.all(np.abs(y[14].cpu().numpy() - ref) <= tol)
    X = dev(np.repeat(x[:, None], 20, 1))
    assert np.all(np.abs(ps.packsell_spmm(A, X).cpu().numpy() - ref[:, None]) <= tol[:, None])
    out = torch.full((csr.n,), -7.0, device="cuda")
    ps.packsell_batch_spmv(ps.packsell_batch_create([A], [dev(x)], [out]))
    assert torch.equal(out, y[14])


@pytest.mark.parametrize("C,variants", [(1, (1, 11, 14)), (32, (1, 4, 9, 13))])
def test_import_is_complete_on_return(C, variants):
    """A matrix imported on one stream may be used on another at once: the
    launch plans are finished when the call returns."""
    need_gpu()
    ps = P()
    rng = np.random.default_rng(C)
    csr = _matrix([int(v) for v in np.minimum(rng.zipf(2.0, 30000), 300)], 5000, seed=5)
    A = ps.packsell_encode_csr(csr, C=C, sigma=1)
    x = dev(I.uniform(csr.m, seed=6))
    blob = ps.packsell_export(A)
    s, t = torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()
    for v in variants:
        ps.packsell_set_spmv_variant(A, v)
        want = ps.packsell_spmv(A, x)
        torch.cuda.synchronize()
        B = ps.packsell_import(blob, stream=s)
        assert s.query()
        ps.packsell_set_spmv_variant(B, v)
        with torch.cuda.stream(t):
            y = ps.packsell_spmv(B, x)
        t.synchronize()
        assert torch.equal(y, want)
