"""The training loss at the ends of the FP32 range: output biases that make some
logits of every row infinite, or so large that a thread's few terms sum past FP32.
The mean loss is then that of FP64: infinite when a target's logit is -inf, and the
sum of the two targets' 2e38 when both have a logit of -2e38 (to FP32 rounding of
each term, 1e-6).  Weights of zero: the logits are the biases."""
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


@pytest.mark.parametrize("bias,want", [(-np.inf, np.inf), (-2e38, 4e38)])
@pytest.mark.parametrize("batch", [64, 192])
def test_loss_at_the_ends_of_the_range(dl, bias, want, batch):
    p, n, h = 16, 64, 64
    params = [np.zeros((h, p)), np.zeros(h), np.zeros((h, h)), np.zeros(h), np.zeros((n, h)), np.zeros(n)]
    params[5][[3, 5]] = bias
    sup = np.tile(np.array([3, 5], np.int32), (batch, 1))  # (two columns of one thread)
    prop = dl.dl_proposer_create(p, n, h, batch, torch.cuda.current_stream())
    dl.dl_proposer_set_weights(prop, params)
    loss = dl.dl_proposer_train(prop, torch.zeros(batch, p, device="cuda"), batch, torch.from_numpy(sup).cuda(), 2,
                                None, batch, 0.0)
    dl.dl_proposer_destroy(prop)
    if np.isinf(want):
        assert loss == want
    else:
        assert abs(loss / want - 1.0) < 1e-6
