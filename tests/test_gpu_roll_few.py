"""The rolled Batch-OMP kernel where its layout changes with the number of signals: one
round of a few warps per SM with all vectors in shared memory, one signal more than
that, and rounds over which the signals are spread evenly.  Bit for bit against the
warp-per-signal kernel (the same arithmetic; no tolerance), which a context made with
DL_OMP_TM=0 codes with."""
import numpy as np
import pytest

from paper_1509_05054_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

# (p, n, s, signals per SM): one to the most warps that hold all vectors in shared memory, and past it
SHAPES = [(36, 129, 9, 1), (64, 256, 16, 14), (64, 256, 16, 15), (64, 256, 10, 16), (64, 256, 10, 17),
          (49, 257, 11, 3), (64, 512, 9, 13), (64, 512, 9, 14), (64, 512, 16, 7), (64, 512, 16, 8),
          (64, 400, 12, 25), (64, 513, 5, 8), (64, 1024, 5, 9), (64, 1024, 8, 7), (64, 1024, 16, 1),
          (100, 1024, 16, 2), (64, 700, 10, 13)]


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


@pytest.mark.parametrize("more", [0, 1])
@pytest.mark.parametrize("p,n,s,per_sm", SHAPES)
def test_layouts_by_number_of_signals(dl, monkeypatch, p, n, s, per_sm, more):
    m = per_sm * torch.cuda.get_device_properties(0).multi_processor_count + more
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
