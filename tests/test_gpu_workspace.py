"""Device memory of a context against the bound that the header states for dl_init, and
the atom update in every form at the shapes where its partial sums take the most of it
(fixed summation order; rows that are no float4 vectors)."""
import numpy as np
import pytest

import oracle
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


def _bound(p, n, m, s):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    per_range = (200 * 1024 - 12 * n - 128) // (4 * p + 16 * s)
    ranges = max(2 * sms, -(-m // per_range))
    return m * (4 * max(-(-n // 32) * 32, p + 3) + 8 * s + 16) + 4 * n * n + 4 * n * (p + 4) * (ranges + 24)


@pytest.mark.parametrize("p,n,m,s", [(64, 512, 1000, 8), (64, 512, 400000, 8), (36, 256, 3000, 6), (49, 200, 5000, 5),
                                     (127, 390, 500, 4), (128, 1024, 2000, 16)])
def test_workspace_within_the_stated_bound(dl, p, n, m, s):
    st = torch.cuda.current_stream()
    dl.dl_destroy(dl.dl_init(p, n, 1, s, dl.DL_FP32, st))  # (the library's own first-use memory)
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    ctx = dl.dl_init(p, n, m, s, dl.DL_FP32, st)
    used = free - torch.cuda.mem_get_info()[0]
    dl.dl_destroy(ctx)
    assert used <= _bound(p, n, m, s) + (24 << 20)  # (about two dozen arrays in 2 MB pages, at the most)


@pytest.mark.parametrize("p,n,m,s,det", [(64, 128, 3001, 5, True), (25, 40, 3001, 4, False), (25, 40, 6001, 4, False),
                                         (127, 1000, 700, 3, False)])
def test_update_with_the_most_partial_sums(dl, p, n, m, s, det):
    g = np.random.default_rng(p)
    Y = g.standard_normal((m, p)).astype(np.float32)
    D = synth.random_dictionary(p, n, seed=9, dtype=np.float32)
    idx = np.sort(np.argsort(g.random((m, n)), axis=1)[:, :s], axis=1).astype(np.int32)
    val = g.standard_normal((m, s)).astype(np.float32)
    cnt = np.full(m, s, np.int32)
    D1, v1, _ = oracle.atom_update(Y.astype(np.float64), D.astype(np.float64), idx, val.astype(np.float64), cnt,
                                   ntilde=None, rule=0)
    ctx = dl.dl_init(p, n, m, s, dl.DL_FP32, torch.cuda.current_stream())
    dl.dl_set_deterministic(ctx, det)
    Dd, v = torch.from_numpy(D.copy()).cuda(), torch.from_numpy(val.reshape(-1)).cuda()
    dl.jau_update(ctx, torch.from_numpy(Y).cuda(), m, Dd, torch.arange(m + 1, device="cuda") * s,
                  torch.from_numpy(idx.reshape(-1)).cuda(), v, None)
    dl.dl_sync(ctx)
    dl.dl_destroy(ctx)
    np.testing.assert_allclose(Dd.cpu().numpy(), D1, rtol=0, atol=1e-5)
    np.testing.assert_allclose(v.cpu().numpy(), v1.reshape(-1), rtol=0, atol=2e-4)
