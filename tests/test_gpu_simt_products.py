"""The CUDA-core products (shapes outside the tensor-core kernel) at the edges of
their tiles: contraction lengths around the 32-column stages, row and atom counts
around the 128-wide tiles, rows that start off a 16-byte boundary.

An FP32 chain of p multiply-adds is within p 2^-24 sum |d_r y_r| of exact (each
of its roundings is relative 2^-24 of a partial sum that |d|.|y| bounds).
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def dl():
    from paper_1509_05054_gb300 import build as _b
    _b.build()
    from paper_1509_05054_gb300 import dl as _dl
    _dl.load()
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    return _dl


@pytest.mark.parametrize("p,n,m,off", [(1, 1, 1, 0), (3, 127, 129, 0), (31, 130, 257, 1), (33, 200, 1000, 3),
                                       (49, 128, 128, 2), (97, 1023, 300, 1), (100, 512, 127, 0),
                                       (127, 257, 385, 0), (128, 64, 5, 0)])
def test_cuda_core_products_at_tile_edges(dl, p, n, m, off):
    g = np.random.default_rng(p * 1000 + n)
    Yh, Dh = g.standard_normal((m, p)).astype(np.float32), g.standard_normal((n, p)).astype(np.float32)
    Y = torch.zeros(m * p + off, device="cuda")[off:].view(m, p)  # off floats from an aligned start
    Y.copy_(torch.from_numpy(Yh))
    D = torch.from_numpy(Dh).cuda()
    A = torch.full((m, n), float("nan"), device="cuda")
    G = torch.full((n, n), float("nan"), device="cuda")
    ctx = dl.dl_init(p, n, m, 1, dl.DL_FP32, torch.cuda.current_stream())
    dl.dl_correlate(ctx, Y, m, D, A)
    dl.dl_gram(ctx, D, G)
    dl.dl_sync(ctx)
    Y64, D64 = Yh.astype(np.float64), Dh.astype(np.float64)
    bound = (p + 1) * 2.0 ** -24
    assert np.all(np.abs(A.cpu().numpy() - Y64 @ D64.T) <= bound * (np.abs(Y64) @ np.abs(D64).T))
    assert np.all(np.abs(G.cpu().numpy() - D64 @ D64.T) <= bound * (np.abs(D64) @ np.abs(D64).T))
    # a coding pass takes both products in one launch: its argmax is that of the product alone
    cp = torch.zeros(m + 1, dtype=torch.int64, device="cuda")
    ri = torch.zeros(m, dtype=torch.int32, device="cuda")
    v = torch.zeros(m, device="cuda")
    dl.omp_code(ctx, Y, m, D, 1, cp, ri, v)
    dl.dl_sync(ctx)
    dl.dl_destroy(ctx)
    if int(cp[m]) == m:
        a = np.abs(A.cpu().numpy())
        chosen = a[np.arange(m), ri.cpu().numpy()]
        assert np.all(chosen >= a.max(axis=1) * (1 - 2.0 ** -17))
