"""The RMSE pairs of several iterations in one call: pair k is written at 2k and
2k + 1 and nowhere else, whatever the number of iterations (from one to more than the
page-locked landing place holds), and equals the pair of the k-th of as many
one-iteration calls.  The fixed summation order makes both the same bits."""
import numpy as np
import pytest

from paper_1509_05054_gb300 import synth

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


@pytest.mark.parametrize("iters", [1, 2, 5, 64, 65])
def test_pairs_of_one_call_and_of_many(dl, iters):
    Y, D, spec = synth.workload_inputs("tiny")
    m, p, n, s = spec["m"], spec["p"], spec["n"], spec["s"]
    Yd = torch.from_numpy(Y).cuda()
    X = (torch.zeros(m + 1, dtype=torch.int64, device="cuda"),
         torch.zeros(m * s, dtype=torch.int32, device="cuda"), torch.zeros(m * s, device="cuda"))
    pairs = []
    for calls, each in ((1, iters), (iters, 1)):
        ctx = dl.dl_init(p, n, m, s, dl.DL_FP32, torch.cuda.current_stream())
        dl.dl_set_deterministic(ctx, True)
        Dd = torch.from_numpy(D.copy()).cuda()
        out = np.full(2 * iters + 2, 7.0)
        for k in range(calls):
            rm = np.zeros(2 * each)
            dl.dl_iterate(ctx, Yd, m, Dd, s, each, *X, rm)
            out[2 * k * each:2 * (k + 1) * each] = rm
        dl.dl_destroy(ctx)
        pairs.append(out)
    np.testing.assert_array_equal(pairs[0], pairs[1])
    assert (pairs[0][:2 * iters] > 0).all() and (pairs[0][:2 * iters] < 1).all()
