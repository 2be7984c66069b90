"""Coefficients of the FP64 re-solve on supports with several near-dependent atoms.

Eight atoms (all of the dictionary), each later one within eps of an earlier one or of
a random direction: Cholesky pivots down to about 10 eps^2.  FP64 Cholesky with
triangular solves has a relative error of a small multiple of 2^-53 / (smallest pivot)
in the coefficients: 7e-9 at eps = 1e-4 (less than the FP32 rounding of the results,
6e-8: together below 1e-7) and 7e-7 at eps = 1e-5, in the oracle as here: 1e-5.

At eps = 1e-5 some orders of selection lead to a last pivot whose exact value lies below
the FP64 rounding of its computation, so that either side may stop one atom short;
those few signals are left out of the comparison.
"""
import numpy as np
import pytest

import oracle

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


def _chain(p, k, eps, g):
    D = []
    for j in range(k):
        if j % 2:
            v = D[-1] + eps * g.standard_normal(p)
        elif j >= 4:
            v = D[j - 3] + eps * g.standard_normal(p)
        else:
            v = g.standard_normal(p)
        D.append(v / np.linalg.norm(v))
    return np.array(D).astype(np.float32)


@pytest.mark.parametrize("eps,tol", [(1e-4, 1e-7), (1e-5, 1e-5)])
@pytest.mark.parametrize("p", [32, 49])
@pytest.mark.parametrize("seed", [0, 1, 2])
def test_coefficients_of_near_dependent_supports(dl, p, eps, tol, seed):
    k = s = 8
    m = 40
    g = np.random.default_rng(seed)
    D = _chain(p, k, eps, g)
    Y = g.standard_normal((m, p)).astype(np.float32)
    ctx = dl.dl_init(p, k, m, s, dl.DL_FP32, torch.cuda.current_stream())
    cp = torch.zeros(m + 1, dtype=torch.int64, device="cuda")
    ri = torch.zeros(m * s, dtype=torch.int32, device="cuda")
    v = torch.zeros(m * s, device="cuda")
    dl.omp_code(ctx, torch.from_numpy(Y).cuda(), m, torch.from_numpy(D).cuda(), s, cp, ri, v)
    dl.dl_sync(ctx)
    listed = dl.dl_last_resolved(ctx)
    dl.dl_destroy(ctx)
    assert listed == m
    idx, val, cnt = csc_to_slots(cp.cpu().numpy(), ri.cpu().numpy(), v.cpu().numpy(), s)
    idx_o, val_o, cnt_o = oracle.omp(Y.astype(np.float64), D.astype(np.float64), s)
    same = (cnt == cnt_o) & (idx == idx_o).all(1)
    assert same.all() if eps > 5e-5 else same.mean() > 0.8
    scale = np.abs(val_o).max(1, keepdims=True)
    assert (np.abs(val - val_o) / scale)[same].max() < tol


@pytest.mark.parametrize("p,n,s,m", [(64, 300, 9, 2000), (49, 130, 10, 700)])
def test_many_listed_signals_with_several_candidates_per_step(dl, p, n, s, m):
    """Every atom has a twin within 1e-6 of it: the two correlations lie inside the FP32
    error of each other at every step, so every signal is listed (more than there are CTAs)
    and the re-solve tells the candidates apart in FP64, as the oracle does."""
    g = np.random.default_rng(n)
    A = g.standard_normal((n // 2, p))
    D = np.vstack([A, A + 1e-6 * np.linalg.norm(A, axis=1, keepdims=True) * g.standard_normal(A.shape) / np.sqrt(p)])
    D = (D / np.linalg.norm(D, axis=1, keepdims=True)).astype(np.float32)[g.permutation(len(D))]
    Y = g.standard_normal((m, p)).astype(np.float32)
    ctx = dl.dl_init(p, len(D), m, s, dl.DL_FP32, torch.cuda.current_stream())
    cp = torch.zeros(m + 1, dtype=torch.int64, device="cuda")
    ri = torch.zeros(m * s, dtype=torch.int32, device="cuda")
    v = torch.zeros(m * s, device="cuda")
    dl.omp_code(ctx, torch.from_numpy(Y).cuda(), m, torch.from_numpy(D).cuda(), s, cp, ri, v)
    dl.dl_sync(ctx)
    listed = dl.dl_last_resolved(ctx)
    dl.dl_destroy(ctx)
    assert listed == m
    idx, val, cnt = csc_to_slots(cp.cpu().numpy(), ri.cpu().numpy(), v.cpu().numpy(), s)
    idx_o, val_o, cnt_o = oracle.omp(Y.astype(np.float64), D.astype(np.float64), s)
    np.testing.assert_array_equal(cnt, cnt_o)
    np.testing.assert_array_equal(idx, idx_o)
    np.testing.assert_allclose(val, val_o, rtol=0, atol=1e-6 * np.abs(val_o).max())
