"""X between slots and CSC at the edges of the kernels' shares: signal counts around
the 256 of a CTA and past the 2048 CTAs of one round, columns of 0 to s entries; and
a caller's CSC that breaks a rule in one column, which stays refused."""
import numpy as np
import pytest

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


@pytest.mark.parametrize("m", [1, 255, 256, 257, 5000, 2048 * 256 + 1, 1300001])
def test_columns_of_identity_coding(dl, m):
    """D = I: signal i with c_i non-zero entries has exactly those as its column."""
    p = n = s = 4
    g = torch.Generator(device="cuda").manual_seed(m)
    on = torch.rand(m, p, generator=g, device="cuda") < 0.5
    mag = 1.0 + torch.rand(m, p, generator=g, device="cuda")
    Y = torch.where(on, mag, torch.zeros_like(mag)).contiguous()
    ctx = dl.dl_init(p, n, m, s, dl.DL_FP32, torch.cuda.current_stream())
    cp = torch.zeros(m + 1, dtype=torch.int64, device="cuda")
    ri = torch.zeros(m * s, dtype=torch.int32, device="cuda")
    v = torch.zeros(m * s, device="cuda")
    dl.omp_code(ctx, Y, m, torch.eye(p, device="cuda"), s, cp, ri, v)
    dl.dl_sync(ctx)
    dl.dl_destroy(ctx)
    want = torch.zeros(m + 1, dtype=torch.int64, device="cuda")
    want[1:] = on.sum(1).cumsum(0)
    assert torch.equal(cp, want)
    nnz = int(want[m])
    assert torch.equal(ri[:nnz].long(), on.nonzero()[:, 1])
    assert torch.allclose(v[:nnz], Y[on], rtol=1e-6, atol=0)


@pytest.mark.parametrize("s", [1, 3, 4, 5, 8, 9, 16])
@pytest.mark.parametrize("fault", ["none", "order", "equal", "low", "high", "long", "back"])
def test_a_column_that_breaks_a_rule_is_refused(dl, s, fault):
    if s == 1 and fault in ("order", "equal"):
        pytest.skip("needs two entries")
    p, n, m = 16, 20, 300
    g = np.random.default_rng(s)
    cols = [np.sort(g.choice(n, size=g.integers(0, s + 1), replace=False)) for _ in range(m)]
    at = 137
    cols[at] = np.sort(g.choice(n, size=s, replace=False))
    cols[at + 1] = np.sort(g.choice(n, size=1, replace=False))
    bad = cols[at].copy()
    if fault == "order":
        bad[-2:] = bad[-2:][::-1]
    elif fault == "equal":
        bad[-1] = bad[-2]
    elif fault == "low":
        bad[0] = -1
    elif fault == "high":
        bad[-1] = n
    cols[at] = bad
    colptr = np.concatenate([[0], np.cumsum([len(c) for c in cols])]).astype(np.int64)
    rowidx = np.concatenate(cols).astype(np.int32)
    if fault == "long":
        colptr[at + 1] += 1  # s + 1 entries, the next column none
    elif fault == "back":
        colptr[at + 1] = colptr[at] - 1
    Y = torch.from_numpy(g.standard_normal((m, p)).astype(np.float32)).cuda()
    D = torch.from_numpy(g.standard_normal((n, p)).astype(np.float32)).cuda()
    val = torch.from_numpy(g.standard_normal(len(rowidx)).astype(np.float32)).cuda()
    ctx = dl.dl_init(p, n, m, s, dl.DL_FP32, torch.cuda.current_stream())
    args = (ctx, Y, m, D, torch.from_numpy(colptr).cuda(), torch.from_numpy(rowidx).cuda(), val, np.zeros(2))
    if fault == "none":
        dl.jau_update(*args)
    else:
        with pytest.raises(dl.DLError) as e:
            dl.jau_update(*args)
        assert e.value.status == dl.DL_EINVAL
    dl.dl_destroy(ctx)
