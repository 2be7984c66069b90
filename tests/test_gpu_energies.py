"""Energies near the top of the FP32 range: ||y||^2 of each signal is finite in FP32,
the sums over a block's or a lane's signals are not.

Four signals (at the places of `rows`) have 1e19 along an axis that no atom has a part
of, and a unit part along an atom of their own; the others are ordinary.  Then
||E||^2 and ||Y||^2 are 4e38 and the atom update is in range: the four atoms turn to that
axis.  RMSE before the update 1 to FP32 rounding of the energies (1e-6); after it the
four errors are FP32 rounding of 1e19 (2^-24 a signal, 1e-5 leaves a wide margin).
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

BIG = 1e19


@pytest.fixture(scope="module")
def dl():
    from paper_1509_05054_gb300 import build as _b
    _b.build()
    from paper_1509_05054_gb300 import dl as _dl
    _dl.load()
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    return _dl


def _problem(p, n, m, rows):
    """D: unit vectors e_0 .. e_{p-2} and random atoms, none with a part along e_{p-1}."""
    g = np.random.default_rng(p)
    D = np.zeros((n, p), np.float32)
    D[:p - 1, :p - 1] = np.eye(p - 1)
    R = g.standard_normal((n - p + 1, p - 1))
    D[p - 1:, :p - 1] = R / np.linalg.norm(R, axis=1, keepdims=True)
    Y = np.zeros((m, p), np.float32)
    Y[:, :p - 1] = 1e-3 * g.standard_normal((m, p - 1))
    for k, i in enumerate(rows):
        Y[i] = 0.0
        Y[i, k], Y[i, p - 1] = 1.0, BIG
    return Y, D


def _check(rm, D, p, rows):
    assert abs(rm[0] - 1.0) < 1e-6 and rm[1] < 1e-5, rm
    axis = np.zeros(p)
    axis[p - 1] = 1.0
    for k in range(len(rows)):
        np.testing.assert_allclose(D[k], axis, rtol=0, atol=1e-5)


@pytest.mark.parametrize("p,n,m,det", [(16, 40, 640, False), (15, 40, 640, False), (16, 40, 3000, True),
                                       (16, 40, 6000, False), (15, 40, 6000, False), (100, 200, 6000, False)])
def test_energies_of_an_update_sum_past_fp32(dl, p, n, m, det):
    s, rows = 1, (0, 1, 2, 3)  # (signals of one block, on different threads)
    Y, D = _problem(p, n, m, rows)
    idx = np.arange(m) % n
    idx[idx < 4] = 4
    idx[list(rows)] = np.arange(4)
    val = Y[np.arange(m), :] @ np.zeros(p, np.float32)
    val[list(rows)] = 1.0
    ctx = dl.dl_init(p, n, m, s, dl.DL_FP32, torch.cuda.current_stream())
    dl.dl_set_deterministic(ctx, det)
    Dd, v, rm = torch.from_numpy(D.copy()).cuda(), torch.from_numpy(val).cuda(), np.zeros(2)
    dl.jau_update(ctx, torch.from_numpy(Y).cuda(), m, Dd, torch.arange(m + 1, device="cuda"),
                  torch.from_numpy(idx.astype(np.int32)).cuda(), v, rm)
    dl.dl_destroy(ctx)
    _check(rm, Dd.cpu().numpy(), p, rows)


def test_energies_of_a_small_problem_sum_past_fp32(dl):
    p, n, m, s = 16, 40, 128, 1
    rows = (0, 32, 64, 96)  # (one warp, so one lane holds the axis of all four)
    Y, D = _problem(p, n, m, rows)
    st = torch.cuda.Stream()
    q = dict(p=p, n=n, s=s, m=m, Y=torch.from_numpy(Y).cuda(), D=torch.from_numpy(D.copy()).cuda(),
             colptr=torch.zeros(m + 1, dtype=torch.int64, device="cuda"),
             rowidx=torch.zeros(m * s, dtype=torch.int32, device="cuda"), val=torch.zeros(m * s, device="cuda"))
    torch.cuda.synchronize()
    b = dl.dl_batch_create([q], autotune=False, stream=st)
    rm = np.zeros(2)
    dl.dl_batch_iterate(b, 1, rm)
    dl.dl_batch_destroy(b)
    _check(rm, q["D"].cpu().numpy(), p, rows)
