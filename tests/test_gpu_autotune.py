"""dl_autotune sets only what the shape's kernels read: a choice that no kernel of the
timed iteration consults keeps its default, so that a later call of another shape or
rule does not run with one that was never measured."""
import numpy as np
import pytest

from paper_1509_05054_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

# (p, n, s, signals per SM, what the iteration reads)
SHAPES = [(36, 128, 4, 34, {"corr_tensor_cores"}),       # several signals per warp, plain update
          (64, 600, 6, 34, {"corr_tensor_cores"}),       # rolled coding kernel, plain update
          (64, 512, 8, 260, set()),                      # residual-form coding, plain update
          (49, 300, 5, 34, {"omp_warps"}),               # CUDA-core products, warp per signal, plain update
          (16, 32, 3, 3, {"corr_tensor_cores", "omp_warps", "accum_mult", "rows_per_sm"})]


@pytest.fixture(scope="module")
def dl():
    from paper_1509_05054_gb300 import build as _b
    _b.build()
    from paper_1509_05054_gb300 import dl as _dl
    _dl.load()
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    return _dl


@pytest.mark.parametrize("p,n,s,per_sm,reads", SHAPES)
def test_choices_that_nothing_reads_keep_their_defaults(dl, monkeypatch, p, n, s, per_sm, reads):
    for name in ("DL_OMP_TM", "DL_OMP_RES", "DL_FORCE_SIMT_GEMM"):
        monkeypatch.delenv(name, raising=False)
    m = per_sm * torch.cuda.get_device_properties(0).multi_processor_count
    Y = torch.from_numpy(np.random.default_rng(p).standard_normal((m, p)).astype(np.float32)).cuda()
    D = torch.from_numpy(synth.random_dictionary(p, n, seed=3, dtype=np.float32)).cuda()
    ctx = dl.dl_init(p, n, m, s, dl.DL_FP32, torch.cuda.current_stream())
    before = dl.dl_get_config(ctx)
    for _ in range(3):
        dl.dl_autotune(ctx, Y, m, D, s)
        after = dl.dl_get_config(ctx)
        assert {k: v for k, v in after.items() if k not in reads} == \
            {k: v for k, v in before.items() if k not in reads}
        assert after["omp_warps"] in (1, 2, 4) and after["accum_mult"] in (1, 2)
        assert after["corr_tensor_cores"] in (0, 1) and after["rows_per_sm"] in (2, 4, 8)
    dl.dl_destroy(ctx)
