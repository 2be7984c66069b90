"""Calls of more iterations than any before them on the same problem.  One-iteration
calls replay a captured iteration from the third on; a longer call needs a longer
array of RMSE pairs, to which a captured iteration must not keep the old address.  The
pairs of the long call equal those of one-iteration calls, bit for bit in the fixed
summation order; the one-iteration calls after it go on right."""
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


@pytest.mark.parametrize("host", [False, True])
@pytest.mark.parametrize("long", [64, 65, 130])
def test_long_call_after_replayed_short_ones(dl, host, long):
    Y, D, spec = synth.workload_inputs("tiny")
    m, p, n, s = spec["m"], spec["p"], spec["n"], spec["s"]
    st = torch.cuda.Stream()
    got = []
    for calls in ([1] * 4 + [long] + [1] * 3, [1] * (long + 7)):
        put = (lambda t: t.pin_memory()) if host else (lambda t: t.cuda())
        Yd, Dd = put(torch.from_numpy(Y)), put(torch.from_numpy(D.copy()))
        X = (put(torch.zeros(m + 1, dtype=torch.int64)), put(torch.zeros(m * s, dtype=torch.int32)),
             put(torch.zeros(m * s)))
        torch.cuda.synchronize()
        ctx = dl.dl_init(p, n, m, s, dl.DL_FP32, st)
        dl.dl_set_deterministic(ctx, True)
        pairs = []
        for k in calls:
            rm = np.zeros(2 * k)
            dl.dl_iterate(ctx, Yd, m, Dd, s, k, *X, rm)
            pairs.append(rm)
        dl.dl_destroy(ctx)
        got.append((np.concatenate(pairs), Dd.cpu().numpy().copy()))
    np.testing.assert_array_equal(got[0][0], got[1][0])
    np.testing.assert_array_equal(got[0][1], got[1][1])
