"""The kernel that codes several signals per warp (small dictionaries, short
supports) against the warp-per-signal kernel: the same arithmetic, so the same bits
(no tolerance).  A context made with DL_OMP_TM=0 codes with the latter.

n at the edges of the lane layouts (1 to 64, 128, 129, 256) and off multiples of
4 (scalar Gram rows), every support length the layouts take, signal counts that
leave the last warp partly empty; among the signals zeros (empty support), exactly
1- and 2-sparse ones (residual stop, while the warp's other signals go on), a
duplicated atom (dependent pivots) and, in half the shapes, exact ties.
"""
import numpy as np
import pytest

from paper_1509_05054_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

MIN = 32 * 152  # fewest signals with n <= 128 on a 152-SM GB300 (half that for n <= 256)
SHAPES = [(4, 5, 1, MIN), (16, 16, 2, MIN + 1), (16, 30, 8, 5003), (25, 63, 5, 6001), (36, 64, 8, 4 * MIN + 3),
          (36, 65, 4, MIN + 2), (49, 101, 6, 7001), (64, 128, 8, 9001), (36, 128, 4, 20001),
          (64, 129, 6, MIN), (49, 200, 5, 2501), (64, 255, 3, 3001), (64, 256, 6, 20003), (121, 256, 1, 2433)]


@pytest.fixture(scope="module")
def dl():
    from paper_1509_05054_gb300 import build as _b
    _b.build()
    from paper_1509_05054_gb300 import dl as _dl
    _dl.load()
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    return _dl


def _code(dl, Y, D, s):
    m, p = Y.shape
    ctx = dl.dl_init(p, D.shape[0], m, s, dl.DL_FP32, torch.cuda.current_stream())
    try:
        cp = torch.zeros(m + 1, dtype=torch.int64, device="cuda")
        ri = torch.zeros(m * s, dtype=torch.int32, device="cuda")
        v = torch.zeros(m * s, device="cuda")
        dl.omp_code(ctx, torch.from_numpy(Y).cuda(), m, torch.from_numpy(D).cuda(), s, cp, ri, v)
        dl.dl_sync(ctx)
        assert dl.dl_last_omp_kernel(ctx) == 0
        return [t.cpu().numpy() for t in (cp, ri, v)] + [dl.dl_last_resolved(ctx)]
    finally:
        dl.dl_destroy(ctx)


@pytest.mark.parametrize("p,n,s,m", SHAPES)
def test_several_signals_per_warp_match_one(dl, monkeypatch, p, n, s, m):
    monkeypatch.setenv("DL_OMP_RES", "0")
    g = np.random.default_rng(n)
    Y = g.standard_normal((m, p)).astype(np.float32)
    D = synth.random_dictionary(p, n, seed=78, dtype=np.float32)
    if n % 2 == 0:  # exact ties: atoms and signals on a coarse grid
        D = (np.round(D * 4) / 4).astype(np.float32)
        D[:, 0] += (np.abs(D).sum(1) == 0)
        Y = np.round(Y * 2).astype(np.float32) / 2
    D[n - 1] = D[0]  # a dependent pair
    for i in range(0, m, 7):
        kind = (i // 7) % 3
        Y[i] = 0.0 if kind == 0 else 3.0 * D[i % n] - (kind - 1) * 2.0 * D[n // 2]
    monkeypatch.delenv("DL_OMP_TM", raising=False)
    new = _code(dl, Y, D, s)
    monkeypatch.setenv("DL_OMP_TM", "0")
    old = _code(dl, Y, D, s)
    for a, b in zip(new, old):
        np.testing.assert_array_equal(a, b)
