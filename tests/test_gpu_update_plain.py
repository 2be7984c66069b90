"""The atom update's three plain passes (errors, bucketed sums, rows) at the edges
of their shapes, against the oracle from an identical X.

Row lengths below, at and between multiples of 32; supports of 1 to 16 with
empty and partial ones among them (four slots are taken at a time); the
fewest signals, whole tiles and one signal past a tile; more pairs per tile than a thread keeps in
registers; an atom that every signal uses (one run of a bucket in every share), atoms
that none does, and the largest dictionary.  Tolerances as for the other update
tests: atoms 1e-5, coefficients 2e-4, RMSE pair 1e-5 and 1e-4.
"""
import numpy as np
import pytest

import oracle
from paper_1509_05054_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

MIN = 32 * 152  # fewest signals that take these passes on a 152-SM GB300
SHAPES = [(4, 8, MIN, 2), (4, 40, MIN + 1, 4), (28, 50, 5003, 5), (32, 64, 4 * MIN + 1, 8), (36, 300, 6001, 9),
          (64, 512, 2 * 64 * 152 + 65, 8), (64, 1024, 5001, 13), (96, 200, 6000, 7), (100, 512, 4999, 12),
          (128, 1024, 5333, 16), (16, 64, 130000, 16),
          (1, 3, MIN, 1), (7, 20, 5001, 3), (25, 64, 6001, 8), (49, 200, 15001, 5), (81, 333, 5000, 12),
          (127, 1023, 4999, 16)]  # rows that are no float4 vectors


@pytest.fixture(scope="module")
def dl():
    from paper_1509_05054_gb300 import build as _b
    _b.build()
    from paper_1509_05054_gb300 import dl as _dl
    _dl.load()
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    return _dl


@pytest.mark.parametrize("rule", [0, 1])
@pytest.mark.parametrize("p,n,m,s", SHAPES)
def test_plain_update_at_its_edges(dl, p, n, m, s, rule):
    g = np.random.default_rng(p + n + m)
    Y = g.standard_normal((m, p)).astype(np.float32)
    D = synth.random_dictionary(p, n, seed=9, dtype=np.float32)
    cnt = g.integers(0, s + 1, m).astype(np.int32)
    cnt[0] = s
    used = n - n // 5  # the last atoms are not used
    idx = np.full((m, s), -1, np.int32)
    for i in range(m):
        c = min(int(cnt[i]), used)
        cnt[i] = c
        if c:
            rest = 1 + g.choice(used - 1, size=c - 1, replace=False) if c > 1 else []
            idx[i, :c] = np.sort(np.concatenate([[0], rest]))  # atom 0: every signal
    val = np.where(idx >= 0, g.standard_normal((m, s)), 0.0).astype(np.float32)
    Y64, D64, v64 = Y.astype(np.float64), D.astype(np.float64), val.astype(np.float64)
    D1, v1, _ = oracle.atom_update(Y64, D64, idx, v64, cnt, ntilde=None, rule=rule)
    colptr = np.concatenate([[0], np.cumsum(cnt)]).astype(np.int64)
    on = idx >= 0
    ctx = dl.dl_init(p, n, m, s, dl.DL_FP32, torch.cuda.current_stream())
    dl.dl_set_update_rule(ctx, rule)
    if n % 50 == 0:  # Y and D one float past a 16-byte boundary
        Yd = torch.zeros(m * p + 1, device="cuda")[1:].view(m, p)
        Yd.copy_(torch.from_numpy(Y))
        Dd = torch.zeros(n * p + 1, device="cuda")[1:].view(n, p)
        Dd.copy_(torch.from_numpy(D))
    else:
        Yd, Dd = torch.from_numpy(Y).cuda(), torch.from_numpy(D.copy()).cuda()
    v = torch.from_numpy(val[on]).cuda()
    rm = np.zeros(2)
    dl.jau_update(ctx, Yd, m, Dd, torch.from_numpy(colptr).cuda(),
                  torch.from_numpy(idx[on]).cuda(), v, rm)
    dl.dl_destroy(ctx)
    np.testing.assert_allclose(Dd.cpu().numpy(), D1, rtol=0, atol=1e-5)
    np.testing.assert_allclose(v.cpu().numpy(), v1[on], rtol=0, atol=2e-4)
    assert abs(rm[0] - oracle.rmse(Y64, D64, idx, v64, cnt)) <= 1e-5
    assert abs(rm[1] - oracle.rmse(Y64, D1, idx, v1, cnt)) <= 1e-4
