"""Which kernels a call launches, by name, on both sides of every line of the dispatch
that results alone do not show: kernels of one group give the same bits or agree to
rounding, so a test that compares them passes as well when one is never taken."""
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


@pytest.fixture(scope="module")
def sms():
    return torch.cuda.get_device_properties(0).multi_processor_count


def _kernels(call):
    """Names of the kernels that call() launches (its second time: the first sets attributes)."""
    call()
    torch.cuda.synchronize()
    activities = [torch.profiler.ProfilerActivity.CUDA]
    for _ in range(3):  # (a process's first trace can come back empty)
        with torch.profiler.profile(activities=activities) as prof:
            torch.zeros(64, device="cuda").add_(1.0)
            call()
            torch.cuda.synchronize()
        names = [e.name for e in prof.events()]
        if any("dlk::" in x or "_kernel" in x for x in names):
            return names
    pytest.skip("no kernel trace on this machine")


def _has(names, kernel):
    return any(kernel + "<" in x or kernel + "(" in x for x in names)


CODE = ("omp_warp_kernel", "omp_sub_kernel", "omp_roll_kernel", "omp_tm_kernel", "romp_kernel")


@pytest.mark.parametrize("p,n,s,per_sm,more,kernel", [
    (36, 128, 4, 32, 0, "omp_sub_kernel"), (36, 128, 4, 32, -1, "omp_warp_kernel"),
    (36, 128, 8, 32, 0, "omp_sub_kernel"), (36, 128, 9, 32, 0, "omp_warp_kernel"),
    (4, 5, 1, 32, 0, "omp_sub_kernel"), (36, 129, 6, 16, 0, "omp_sub_kernel"),
    (36, 129, 6, 16, -1, "omp_warp_kernel"), (36, 256, 7, 33, 0, "omp_warp_kernel"),
    (36, 257, 6, 33, 0, "omp_warp_kernel"), (36, 129, 9, 1, 0, "omp_roll_kernel"),
    (64, 513, 5, 1, 0, "omp_roll_kernel"), (64, 513, 4, 1, 0, "omp_warp_kernel"),
    (64, 512, 8, 4, 0, "omp_tm_kernel"), (64, 512, 8, 192, 0, "romp_kernel")])
def test_coding_kernel(dl, monkeypatch, sms, p, n, s, per_sm, more, kernel):
    for name in ("DL_OMP_TM", "DL_OMP_RES"):
        monkeypatch.delenv(name, raising=False)
    m = per_sm * sms + more
    Y = torch.from_numpy(np.random.default_rng(p).standard_normal((m, p)).astype(np.float32)).cuda()
    D = torch.from_numpy(synth.random_dictionary(p, n, seed=3, dtype=np.float32)).cuda()
    X = (torch.zeros(m + 1, dtype=torch.int64, device="cuda"),
         torch.zeros(m * s, dtype=torch.int32, device="cuda"), torch.zeros(m * s, device="cuda"))
    ctx = dl.dl_init(p, n, m, s, dl.DL_FP32, torch.cuda.current_stream())
    names = _kernels(lambda: dl.omp_code(ctx, Y, m, D, s, *X))
    dl.dl_destroy(ctx)
    assert [k for k in CODE if _has(names, k)] == [kernel]


UPDATE = ("errors_kernel", "sums_kernel", "rows_plain_kernel", "accum4_kernel", "accum_kernel", "accum_det_kernel",
          "rows4_kernel", "rows_kernel", "pad_atoms_kernel")
PLAIN = {"errors_kernel", "sums_kernel", "rows_plain_kernel"}


@pytest.mark.parametrize("p,per_sm,more,det,kernels", [
    (64, 32, 0, False, PLAIN), (64, 32, -1, False, {"accum4_kernel", "rows4_kernel"}),
    (49, 32, 0, False, PLAIN | {"pad_atoms_kernel"}), (49, 32, -1, False, {"accum_kernel", "rows_kernel"}),
    (64, 33, 0, True, {"accum_det_kernel", "rows4_kernel"}), (128, 32, 0, False, PLAIN)])
def test_update_kernels(dl, sms, p, per_sm, more, det, kernels):
    n, s, m = 200, 3, per_sm * sms + more
    g = np.random.default_rng(p)
    Y = torch.from_numpy(g.standard_normal((m, p)).astype(np.float32)).cuda()
    D = torch.from_numpy(synth.random_dictionary(p, n, seed=3, dtype=np.float32)).cuda()
    idx = np.sort(np.argsort(g.random((m, n)), axis=1)[:, :s], axis=1).astype(np.int32)
    ri, v = torch.from_numpy(idx.reshape(-1)).cuda(), torch.ones(m * s, device="cuda")
    cp = torch.arange(m + 1, device="cuda") * s
    ctx = dl.dl_init(p, n, m, s, dl.DL_FP32, torch.cuda.current_stream())
    dl.dl_set_deterministic(ctx, det)
    names = _kernels(lambda: dl.jau_update(ctx, Y, m, D, cp, ri, v, None))
    dl.dl_destroy(ctx)
    assert {k for k in UPDATE if _has(names, k)} == kernels
