"""Signals of every kind side by side in one warp of the kernel that codes several
signals per warp: live ones, zero ones, ones with a NaN or an infinity, ones whose
correlations tie exactly (the masked correlation lies among those that the other lanes
read to find the selected atom), 1-sparse ones that stop at once.

The finite signals' supports and coefficients are those of the warp-per-signal
kernel bit for bit (the same arithmetic); the ties go to the lowest atom; a
non-finite signal has an empty column and the call reports it.  The small-problem
batch runs the same loop: its supports are those of the oracle.
"""
import numpy as np
import pytest

import oracle
from paper_1509_05054_gb300 import synth

from _common import csc_to_slots

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


def _signals(D, m, g):
    """Kinds by turns, so that the two or four signals of a warp differ."""
    n, p = D.shape
    Y = g.standard_normal((m, p)).astype(np.float32)
    kind = g.integers(0, 6, m)
    Y[kind == 1] = 0.0
    Y[kind == 2, 0] = np.nan
    Y[kind == 3, p - 1] = np.inf
    tie = np.flatnonzero(kind == 4)
    a, b = g.integers(0, p, (2, len(tie)))  # D starts with the unit vectors: |y_a| = |y_b|
    Y[tie] = 0.0
    Y[tie, a] = 2.0
    Y[tie, b] = -2.0
    other = np.abs(Y[tie] @ D[p:].T).max(1)
    kind[tie[other > 1.9]] = 5  # (another atom correlates as much)
    one = np.flatnonzero(kind == 5)
    Y[one] = 3.0 * D[g.integers(0, n, len(one))]
    return Y, kind


def _code(dl, Y, D, s):
    m, p = Y.shape
    ctx = dl.dl_init(p, D.shape[0], m, s, dl.DL_FP32, torch.cuda.current_stream())
    try:
        cp = torch.zeros(m + 1, dtype=torch.int64, device="cuda")
        ri = torch.zeros(m * s, dtype=torch.int32, device="cuda")
        v = torch.zeros(m * s, device="cuda")
        dl.omp_code(ctx, torch.from_numpy(Y).cuda(), m, torch.from_numpy(D).cuda(), s, cp, ri, v)
        with pytest.raises(dl.DLError) as e:
            dl.dl_sync(ctx)
        assert e.value.status == dl.DL_ENUMERIC
        return csc_to_slots(cp.cpu().numpy(), ri.cpu().numpy(), v.cpu().numpy(), s)
    finally:
        dl.dl_destroy(ctx)


@pytest.mark.parametrize("p,n,s", [(16, 40, 4), (36, 128, 5), (49, 200, 6)])
def test_kinds_of_signals_side_by_side(dl, monkeypatch, p, n, s):
    monkeypatch.setenv("DL_OMP_RES", "0")
    m = 33 * torch.cuda.get_device_properties(0).multi_processor_count + 1
    g = np.random.default_rng(p)
    D = np.vstack([np.eye(p), synth.random_dictionary(p, n - p, seed=5, dtype=np.float64)]).astype(np.float32)
    Y, kind = _signals(D, m, g)
    monkeypatch.delenv("DL_OMP_TM", raising=False)
    idx, val, cnt = _code(dl, Y, D, s)
    monkeypatch.setenv("DL_OMP_TM", "0")
    idx0, val0, cnt0 = _code(dl, Y, D, s)
    np.testing.assert_array_equal(cnt, cnt0)
    np.testing.assert_array_equal(idx, idx0)
    np.testing.assert_array_equal(val, val0)
    assert not cnt[(kind == 1) | (kind == 2) | (kind == 3)].any()
    tie = np.flatnonzero(kind == 4)
    assert len(tie) > m // 20
    for i in tie:
        assert list(idx[i, :cnt[i]]) == list(np.flatnonzero(Y[i]))  # (1-sparse where both fell on one atom)


def test_kinds_of_signals_side_by_side_in_a_batch(dl):
    p, n, s, m = 16, 40, 4, 203
    g = np.random.default_rng(2)
    D = np.vstack([np.eye(p), synth.random_dictionary(p, n - p, seed=5, dtype=np.float64)]).astype(np.float32)
    Y, kind = _signals(D, m, g)
    Y[(kind == 2) | (kind == 3)] = 0.0
    st = torch.cuda.Stream()
    q = dict(p=p, n=n, s=s, m=m, Y=torch.from_numpy(Y).cuda(), D=torch.from_numpy(D.copy()).cuda(),
             colptr=torch.zeros(m + 1, dtype=torch.int64, device="cuda"),
             rowidx=torch.zeros(m * s, dtype=torch.int32, device="cuda"), val=torch.zeros(m * s, device="cuda"))
    torch.cuda.synchronize()
    b = dl.dl_batch_create([q], autotune=False, stream=st)
    dl.dl_batch_iterate(b, 1, np.zeros(2))
    dl.dl_batch_destroy(b)
    idx, _, cnt = csc_to_slots(q["colptr"].cpu().numpy(), q["rowidx"].cpu().numpy(), q["val"].cpu().numpy(), s)
    idx_o, _, cnt_o = oracle.omp(Y.astype(np.float64), D.astype(np.float64), s)
    exact = kind != 5  # (how long an exactly 1-sparse signal goes on is rounding)
    np.testing.assert_array_equal(cnt[exact], cnt_o[exact])
    np.testing.assert_array_equal(idx[exact], idx_o[exact])
