"""The proposer's products at the edges of their tiles: widths of one, two and a
half, and several 128-column tiles, a padded signal length, batches below one row
tile and ones whose contraction does not divide into equal slices.

Gradients of the last batch and the mean loss against the FP64 network on the
same BF16-rounded weights and inputs.  Each of up to five chained BF16 roundings
(activations, dZ, dA) is relative 2^-9 per element and independent: 2e-2 in the
Frobenius norm leaves a factor of four.
"""
import numpy as np
import pytest

from oracle import mlp
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


def _bf16(a):
    return torch.from_numpy(np.asarray(a, np.float32)).to(torch.bfloat16).to(torch.float64).numpy()


def _rel(a, b):
    return float(np.linalg.norm(a - b) / max(np.linalg.norm(b), 1e-30))


@pytest.mark.parametrize("p,n,h,batch,m,permuted", [(16, 64, 64, 64, 200, False), (100, 320, 192, 320, 960, True),
                                                    (64, 576, 640, 576, 1152, False),
                                                    (121, 1024, 128, 192, 192, True)])
def test_gradients_and_logits_at_tile_edges(dl, p, n, h, batch, m, permuted):
    g = np.random.default_rng(p)
    params = synth.proposer_init(p, n, h, seed=2, positives=5)
    Y = g.standard_normal((m, p)).astype(np.float32)
    s = 5
    sup = np.sort(np.argsort(g.random((m, n)), axis=1)[:, :s], axis=1).astype(np.int32)
    sup[::7, s - 1] = -1  # an empty slot
    perm = g.permutation(m) if permuted else np.arange(m)
    prop = dl.dl_proposer_create(p, n, h, batch, torch.cuda.current_stream())
    dl.dl_proposer_set_weights(prop, params)
    Yd = torch.from_numpy(Y).cuda()
    loss = dl.dl_proposer_train(prop, Yd, m, torch.from_numpy(sup).cuda(), s,
                                torch.from_numpy(perm).cuda() if permuted else None, batch, 0.0)
    grads = dl.dl_proposer_get(prop, 1, [w.shape for w in params])
    logits = torch.zeros(m, n, device="cuda")
    cand = torch.zeros(m, 8, dtype=torch.int32, device="cuda")
    cand2 = torch.zeros_like(cand)
    dl.dl_proposer_forward(prop, Yd, m, logits=logits, cand=cand, K=8)
    dl.dl_proposer_forward(prop, Yd, m, cand=cand2, K=8)
    dl.dl_proposer_destroy(prop)
    pb = [_bf16(w) if w.ndim == 2 else w for w in params]
    losses = []
    for r0 in range(0, m - batch + 1, batch):
        rows = perm[r0:r0 + batch]
        T = np.zeros((batch, n))
        for i, r in enumerate(rows):
            T[i, sup[r][sup[r] >= 0]] = 1.0
        z, cache = mlp.forward(pb, _bf16(Y[rows]))
        losses.append(mlp.loss(z, T))
    ref = mlp.backward(pb, cache, z, T)
    assert abs(loss - np.mean(losses)) < 1e-2 * np.mean(losses)
    for k, (gk, rk) in enumerate(zip(grads, ref)):
        assert _rel(gk, rk) < 2e-2, (k, _rel(gk, rk))
    z_all, _ = mlp.forward(pb, _bf16(Y))
    assert _rel(logits.cpu().numpy(), z_all) < 2e-2
    assert torch.equal(cand, cand2)
