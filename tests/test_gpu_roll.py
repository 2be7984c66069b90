"""The rolled Batch-OMP kernel (long supports, wide dictionaries) and the FP64
re-solve at the edges of their shapes.

The rolled kernel does the arithmetic of the warp-per-signal kernel operation
by operation, so the two must agree bit for bit (no tolerance): a context made
with DL_OMP_TM=0 codes with the latter.  Shapes: the smallest and largest n of
each vector length (129, 256, 257, 512, 513, 1024), supports where the vectors
fit in tensor memory alone, where the last few go to shared memory, and where
fewer warps are resident, one signal, and counts that leave the last round of
warps ragged.  Among the signals: zeros (empty support), exactly 1- and 2-sparse
ones (residual stop) and, through a duplicated atom, dependent pivots.
"""
import numpy as np
import pytest

import oracle
from paper_1509_05054_gb300 import synth

from _common import csc_to_slots

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

SHAPES = [(64, 1024, 5, 700), (64, 1024, 8, 2500), (64, 513, 9, 333), (64, 1024, 10, 1900),
          (100, 700, 12, 257), (36, 1024, 16, 300), (64, 512, 9, 4000), (49, 257, 11, 517),
          (64, 400, 14, 129), (64, 512, 16, 300), (64, 129, 9, 1000), (64, 256, 16, 5001),
          (100, 256, 12, 1)]


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
        return [t.cpu().numpy() for t in (cp, ri, v)], dl.dl_last_omp_kernel(ctx), dl.dl_last_resolved(ctx)
    finally:
        dl.dl_destroy(ctx)


@pytest.mark.parametrize("p,n,s,m", SHAPES)
def test_rolled_kernel_matches_warp_kernel_bit_for_bit(dl, monkeypatch, p, n, s, m):
    Y = synth.image_patches(m, side=int(np.sqrt(p)), workload_id=77).astype(np.float32)
    D = synth.random_dictionary(p, n, seed=78, dtype=np.float32)
    D[n - 1] = D[0]  # a dependent pair
    for i in range(0, m, 41):
        kind = (i // 41) % 3
        Y[i] = 0.0 if kind == 0 else 3.0 * D[1 + i % (n - 2)] - (kind - 1) * 2.0 * D[n // 2]
    monkeypatch.delenv("DL_OMP_TM", raising=False)
    rolled, kind, res = _code(dl, Y, D, s)
    monkeypatch.setenv("DL_OMP_TM", "0")
    warp, kind0, res0 = _code(dl, Y, D, s)
    assert kind == 1 and kind0 == 0
    assert res == res0
    for a, b in zip(rolled, warp):
        np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("p", [3, 33, 100, 128])
def test_resolve_matches_oracle_on_near_dependent_pairs(dl, p):
    """Atoms e_{p-1} and ~ e_{p-1} + 5e-4 e_{p-2}: an FP32 pivot of 2.5e-7, listed for the FP64
    re-solve, which finds both (coefficients to FP32 rounding of values up to 2e4: rtol 1e-5)."""
    E = np.eye(p)
    b = E[p - 1] + 5e-4 * E[p - 2]
    D = np.vstack([E[:p - 2], E[p - 1], b / np.linalg.norm(b)]).astype(np.float32)
    s, m = min(3, p), 50
    g = np.random.default_rng(5)
    Y = np.zeros((m, p), np.float32)
    Y[:, p - 1], Y[:, p - 2] = 2.0, 10.0
    Y[:, 0] += (g.standard_normal(m) * 0.5).astype(np.float32) if p > 3 else 0.0
    (cp, ri, v), _, nres = _code(dl, Y, D, s)
    idx, val, cnt = csc_to_slots(cp, ri, v, s)
    idx_o, val_o, cnt_o = oracle.omp(Y.astype(np.float64), D.astype(np.float64), s)
    assert nres == m
    np.testing.assert_array_equal(cnt, cnt_o)
    np.testing.assert_array_equal(idx, idx_o)
    np.testing.assert_allclose(val, val_o, rtol=1e-5, atol=1e-6)
