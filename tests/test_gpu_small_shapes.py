"""The one-launch batch of small problems at the edges of its layout, against a
context of its own per problem.

With an odd p both take the correlations as the same FP32 chains, so the supports
agree exactly; atoms and coefficients differ by the order of FP32 sums (1e-5, as
in the other update tests).  Shapes: the largest (whose coding state leaves room for
fewer warps), the smallest, supports of 1 to 8, signal counts that leave a warp's
four signals partly empty; zero signals and a dependent pair among the inputs.
"""
import numpy as np
import pytest

from paper_1509_05054_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

SHAPES = [(31, 64, 8, 701), (31, 64, 6, 130), (21, 50, 5, 333), (7, 9, 3, 1), (1, 1, 1, 6), (29, 33, 4, 1500),
          (9, 63, 7, 64)]


@pytest.fixture(scope="module")
def dl():
    from paper_1509_05054_gb300 import build as _b
    _b.build()
    from paper_1509_05054_gb300 import dl as _dl
    _dl.load()
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    return _dl


def test_batch_matches_contexts_of_their_own(dl):
    probs, alone = [], []
    st = torch.cuda.Stream()
    for k, (p, n, s, m) in enumerate(SHAPES):
        g = np.random.default_rng(k)
        D = synth.random_dictionary(p, n, seed=k, dtype=np.float32)
        if n > 2:
            D[n - 1] = D[0]
        Y = g.standard_normal((m, p)).astype(np.float32)
        Y[::5] = 0.0
        for out in (probs, alone):
            out.append(dict(p=p, n=n, s=s, m=m, Y=torch.from_numpy(Y).cuda(), D=torch.from_numpy(D.copy()).cuda(),
                            colptr=torch.zeros(m + 1, dtype=torch.int64, device="cuda"),
                            rowidx=torch.zeros(m * s, dtype=torch.int32, device="cuda"),
                            val=torch.zeros(m * s, device="cuda")))
    torch.cuda.synchronize()
    batch = dl.dl_batch_create(probs, autotune=False, stream=st)
    rm = np.zeros(2 * len(SHAPES))
    dl.dl_batch_iterate(batch, 1, rm)
    dl.dl_batch_destroy(batch)
    for k, (b, a) in enumerate(zip(probs, alone)):
        ctx = dl.dl_init(a["p"], a["n"], a["m"], a["s"], dl.DL_FP32, st)
        r1 = np.zeros(2)
        dl.dl_iterate(ctx, a["Y"], a["m"], a["D"], a["s"], 1, a["colptr"], a["rowidx"], a["val"], r1)
        dl.dl_destroy(ctx)
        assert torch.equal(b["colptr"], a["colptr"]), SHAPES[k]
        nnz = int(a["colptr"][-1])
        assert torch.equal(b["rowidx"][:nnz], a["rowidx"][:nnz]), SHAPES[k]
        np.testing.assert_allclose(b["D"].cpu(), a["D"].cpu(), rtol=0, atol=1e-5)
        np.testing.assert_allclose(b["val"][:nnz].cpu(), a["val"][:nnz].cpu(), rtol=0, atol=2e-4)
        np.testing.assert_allclose(rm[2 * k:2 * k + 2], r1, rtol=0, atol=1e-5)
