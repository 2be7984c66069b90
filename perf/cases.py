"""Timed cases: what a user of the library has it do, through its public calls.

A case names one call on one problem: a whole dictionary-learning iteration
(``dl_iterate``), sparse coding alone (``omp_code``), the atom update alone
(``jau_update``), an iteration from host buffers, a batch of small problems
(``dl_batch_iterate``) or the training pass of the support proposer
(``dl_proposer_train``).  Sizes are those of the workloads in
``paper_1509_05054_gb300.synth`` and of the tests, and between them.

Signals are made on the GPU from the seed: patches of 1/f^2 random fields
(mean removed, unit variance) for the image-patch problems, noisy sparse
combinations of a hidden dictionary for the recovery problems.  A pass starts
from the dictionary at hand, so it first copies that into the buffer which the
iteration updates in place.
"""
import math

import numpy as np
import torch

from paper_1509_05054_gb300 import dl, synth

PRECISIONS = {"fp32": dl.DL_FP32, "bf16": dl.DL_BF16, "fp8": dl.DL_FP8}


def listed():
    return [
        # the smallest call: one tracked iteration of a toy recovery problem
        # (the repository's "tiny"), bound by launches and host latency
        dict(name="recovery_tiny", kind="iterate", data="recovery", p=16, n=32, m=1000, s=3,
             precision="fp32", track=True),
        # dictionary recovery (the paper's Table 1): 200 small problems at once
        dict(name="recovery_batch", kind="batch", data="recovery", count=200, p=20, n=50, m=1500, s=4),
        # 8x8 image patches, a 4x overcomplete dictionary, a moderate training set
        dict(name="patch_n256", kind="iterate", data="patch", p=64, n=256, m=20000, s=6,
             precision="fp32", track=False),
        # the throughput workload: 8x overcomplete, 1e5 patches
        dict(name="patch_n512", kind="iterate", data="patch", p=64, n=512, m=100000, s=8,
             precision="fp32", track=False),
        # the same with BF16 correlations
        dict(name="patch_n512_bf16", kind="iterate", data="patch", p=64, n=512, m=100000, s=8,
             precision="bf16", track=False),
        # the largest dictionary: 16x overcomplete, longer supports
        dict(name="patch_n1024", kind="iterate", data="patch", p=64, n=1024, m=46000, s=10,
             precision="fp32", track=False),
        # 10x10 patches with long supports
        dict(name="patch10_n512", kind="iterate", data="patch", p=100, n=512, m=30000, s=12,
             precision="fp32", track=False),
        # odd sizes: 7x7 patches (rows of 49 floats), n no multiple of 32, a ragged signal count
        dict(name="patch7_odd", kind="iterate", data="patch", p=49, n=200, m=15001, s=5,
             precision="fp32", track=False),
        # coding alone with a dictionary at hand: 6x6 patches, short supports
        dict(name="encode_patch6", kind="encode", data="patch", p=36, n=128, m=60000, s=4,
             precision="fp32"),
        # the atom update alone, from the caller's own sparse representation
        dict(name="update_n512", kind="update", data="patch", p=64, n=512, m=100000, s=8,
             precision="fp32"),
        # the throughput workload with everything in page-locked host memory
        dict(name="host_n512", kind="host", data="patch", p=64, n=512, m=100000, s=8,
             precision="fp32"),
        # training the support proposer: forward, backward and gradients of 16 batches
        dict(name="proposer_train", kind="train", p=64, n=512, hidden=512, m=65536, s=8, batch=4096),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["iterate", "iterate", "iterate", "encode", "update", "host", "batch", "train"])
    if kind == "batch":
        p, s = rng.randint(12, 32), rng.randint(2, 6)
        return dict(kind=kind, data="recovery", count=_log(rng, 8, 200), p=p, n=rng.randint(p, 64),
                    m=_log(rng, 200, 1500), s=s)
    if kind == "train":
        batch = rng.choice([256, 512, 1024, 2048, 4096])
        return dict(kind=kind, p=rng.choice([16, 36, 64, 100]), n=rng.choice([128, 256, 512]),
                    hidden=rng.choice([128, 256, 512]), m=batch * rng.randint(2, 16) + rng.randint(0, 200),
                    s=rng.randint(3, 8), batch=batch)
    if kind == "iterate" and rng.random() < 0.25:  # recovery problems
        p = rng.randint(8, 32)
        return dict(kind=kind, data="recovery", p=p, n=rng.randint(p, 4 * p), m=_log(rng, 500, 20000),
                    s=rng.randint(2, 5), precision="fp32", track=rng.random() < 0.5)
    side = rng.randint(4, 11)
    p = side * side
    n = min(1024, max(p, _log(rng, 64, 1024)))
    if rng.random() < 0.5:
        n = max(64, (n + 32) // 64 * 64)
    s = rng.randint(3, min(12, p // 4))
    # no more work than the throughput workload or the largest dictionary
    most = 4.0e9 / (n * (2 * p + s * s))
    case = dict(kind=kind, data="patch", p=p, n=n, m=min(_log(rng, 1000, 100000), int(most)), s=s,
                precision=rng.choice(["fp32", "fp32", "fp32", "bf16", "fp8"]) if kind == "iterate" else "fp32")
    if kind == "iterate":
        case["track"] = rng.random() < 0.25
    return case


# ---- inputs --------------------------------------------------------------------

def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _patches(m, side, gen):
    """m mean-removed, unit-variance side x side patches of 1/f^2 random fields, (m, side^2) float32."""
    size = synth.IMAGE_SIZE
    images = -(-m // synth.PATCHES_PER_IMAGE)
    f = torch.fft.fftfreq(size, device="cuda", dtype=torch.float64)
    f = torch.sqrt(f[:, None] ** 2 + f[None, :] ** 2)
    amp = torch.where(f > 0, 1.0 / f.clamp(min=1e-9), torch.zeros_like(f))
    out = []
    for _ in range(images):
        white = torch.randn(size, size, generator=gen, device="cuda", dtype=torch.float64)
        image = torch.fft.ifft2(torch.fft.fft2(white) * amp).real
        r = torch.randint(0, size - side + 1, (synth.PATCHES_PER_IMAGE,), generator=gen, device="cuda")
        c = torch.randint(0, size - side + 1, (synth.PATCHES_PER_IMAGE,), generator=gen, device="cuda")
        a = torch.arange(side, device="cuda")
        P = image[r[:, None, None] + a[None, :, None], c[:, None, None] + a[None, None, :]].reshape(-1, side * side)
        P = P - P.mean(1, keepdim=True)
        out.append(P / P.square().mean(1, keepdim=True).sqrt())
    return torch.cat(out)[:m].float().contiguous()


def _unit(D):
    return D / D.norm(dim=-1, keepdim=True)


def _recovery(count, p, n, m, s, gen):
    """count problems: Y (count, m, p) of s atoms of a hidden dictionary each, N(0,1) weights,
    30 dB noise, and a starting dictionary of normalised signals (count, n, p); float32."""
    D0 = _unit(torch.randn(count, n, p, generator=gen, device="cuda", dtype=torch.float64))
    at = torch.rand(count, m, n, generator=gen, device="cuda").topk(s, dim=-1).indices
    w = torch.randn(count, m, s, generator=gen, device="cuda", dtype=torch.float64)
    X = torch.zeros(count, m, n, device="cuda", dtype=torch.float64).scatter_(2, at, w)
    Y = X @ D0
    Y = Y + Y.square().mean().sqrt() * 10.0 ** (-30.0 / 20.0) * torch.randn(
        Y.shape, generator=gen, device="cuda", dtype=torch.float64)
    return Y.float().contiguous(), _unit(Y[:, :n]).float().contiguous()


def _inputs(case, seed):
    """(Y, D) of the case's problem or problems, (count, m, p) and (count, n, p) float32 on the GPU."""
    gen = _generator(seed)
    p, n, m, s = case["p"], case["n"], case["m"], case["s"]
    if case["data"] == "recovery":
        return _recovery(case.get("count", 1), p, n, m, s, gen)
    Y = _patches(m, int(math.isqrt(p)), gen)
    D = _unit(torch.randn(n, p, generator=gen, device="cuda", dtype=torch.float64)).float()
    return Y[None], D[None]


def _given_x(Y, D, s):
    """A sparse representation that a program of its own might bring to the atom update: the s
    atoms of largest |D y| of each signal, with ridge-regularised least-squares coefficients."""
    idx = (Y @ D.T).abs().topk(s, dim=1).indices.sort(dim=1).values
    A = D.double()[idx]
    G = A @ A.transpose(1, 2) + 1e-2 * torch.eye(s, device="cuda", dtype=torch.float64)
    x = torch.linalg.solve(G, A @ Y.double()[:, :, None])[:, :, 0]
    return idx, x.float()


class _Batch:
    """A dl_batch handle, freed with the state that holds it."""

    def __init__(self, problems, stream):
        self.handle = dl.dl_batch_create(problems, autotune=False, stream=stream)

    def __del__(self):
        dl.dl_batch_destroy(self.handle)


class _Proposer:
    """A dl_proposer handle, freed with the state that holds it."""

    def __init__(self, case, stream):
        self.handle = dl.dl_proposer_create(case["p"], case["n"], case["hidden"], case["batch"], stream)

    def __del__(self):
        dl.dl_proposer_destroy(self.handle)


def _csc(m, s, **where):
    return (torch.zeros(m + 1, dtype=torch.int64, **where), torch.zeros(m * s, dtype=torch.int32, **where),
            torch.zeros(m * s, dtype=torch.float32, **where))


def _train_inputs(case, seed):
    p, n, h, s = case["p"], case["n"], case["hidden"], case["s"]
    gen = _generator(seed)
    Y = _patches(case["m"], int(math.isqrt(p)), gen)
    sup = torch.rand(case["m"], n, generator=gen, device="cuda").topk(s, dim=1).indices.sort(dim=1).values.int()
    return Y, sup.contiguous(), synth.proposer_init(p, n, h, seed=seed, positives=s)


def prepare(case, seed):
    kind = case["kind"]
    stream = torch.cuda.Stream()
    state = dict(case=case, stream=stream)
    if kind == "train":
        Y, sup, weights = _train_inputs(case, seed)
        prop = _Proposer(case, stream)
        torch.cuda.synchronize()
        dl.dl_proposer_set_weights(prop.handle, weights)
        return dict(state, Y=Y, sup=sup, prop=prop, shapes=[w.shape for w in weights])
    Y, D = _inputs(case, seed)
    s = case["s"]
    count, m, p = Y.shape
    n = D.shape[1]
    if kind == "batch":
        work = D.clone()
        X = [x.repeat(count, 1) for x in _csc(m, s, device="cuda")]
        problems = [dict(p=p, n=n, m=m, s=s, Y=Y[k], D=work[k], colptr=X[0][k], rowidx=X[1][k], val=X[2][k])
                    for k in range(count)]
        torch.cuda.synchronize()
        batch = _Batch(problems, stream)
        work.copy_(D)
        return dict(state, Y=Y, D0=D, D=work, X=X, batch=batch)
    ctx = dl.Context(p, n, m, s, PRECISIONS[case["precision"]], stream=stream)
    state.update(ctx=ctx, m=m, D0=D[0].contiguous())
    if kind == "host":
        pin = dict(pin_memory=True)
        colptr, rowidx, val = _csc(m, s, **pin)
        return dict(state, Y=Y[0].cpu().pin_memory(), D0=D[0].cpu(), D=torch.empty(n, p, **pin),
                    colptr=colptr, rowidx=rowidx, val=val)
    colptr, rowidx, val = _csc(m, s, device="cuda")
    if kind == "update":
        idx, x = _given_x(Y[0], D[0], s)
        colptr = torch.arange(m + 1, device="cuda", dtype=torch.int64) * s
        rowidx, val = idx.int().reshape(-1).contiguous(), x.reshape(-1).contiguous()
    return dict(state, Y=Y[0].contiguous(), D=D[0].clone(), colptr=colptr, rowidx=rowidx, val=val)


def run(state):
    case, kind = state["case"], state["case"]["kind"]
    if kind == "train":  # gradients of the last batch and the mean loss of the pass
        prop = state["prop"].handle
        loss = dl.dl_proposer_train(prop, state["Y"], case["m"], state["sup"], case["s"],
                                    batch=case["batch"], lr=0.0)
        return dict(loss=loss, grad=dl.dl_proposer_get(prop, 1, state["shapes"]))
    if kind == "batch":
        with torch.cuda.stream(state["stream"]):
            state["D"].copy_(state["D0"])
        dl.dl_batch_iterate(state["batch"].handle, 1)
        colptr, rowidx, val = state["X"]
        return dict(D=state["D"], colptr=colptr, rowidx=rowidx, val=val)
    ctx, m, s = state["ctx"].ctx, state["m"], case["s"]
    Y, D, X = state["Y"], state["D"], (state["colptr"], state["rowidx"], state["val"])
    out = dict(colptr=X[0], rowidx=X[1], val=X[2])
    if kind == "encode":
        dl.omp_code(ctx, Y, m, D, s, *X)
        return out
    if kind == "update":
        dl.jau_update(ctx, Y, m, D, *X)
        return dict(out, D=D)
    if kind == "host":
        D.copy_(state["D0"])
        dl.dl_iterate(ctx, Y, m, D, s, 1, *X)
        return dict(out, D=D)
    with torch.cuda.stream(state["stream"]):
        D.copy_(state["D0"])
    if case["track"]:
        rmse = np.zeros(2)
        dl.dl_iterate(ctx, Y, m, D, s, 1, *X, rmse)
        return dict(out, D=D, rmse=[float(v) for v in rmse])
    dl.dl_iterate(ctx, Y, m, D, s, 1, *X)
    return dict(out, D=D)


def work(case):
    """Bytes: signals and dictionary read once, results written once.  Operations: one product of the
    signals with the dictionary and Batch-OMP's updates of the correlations; errors, atom sums and
    coefficients of the update; the proposer's three products, forward and both backward ones."""
    p, n, m, s = case["p"], case["n"], case["m"], case["s"]
    if case["kind"] == "train":
        h = case["hidden"]
        weights = p * h + h * h + h * n
        return dict(bytes=4 * m * (p + s) + 8 * weights, flops=m * (6 * weights - 2 * p * h))
    count = case.get("count", 1)
    code = 2 * n * p + n * s * (s - 1)
    update = 10 * s * p
    flops = count * m * {"encode": code, "update": update}.get(case["kind"], code + update)
    moved = 4 * m * p + 8 * m * s + 8 * (m + 1) + 4 * n * p
    if case["kind"] != "encode":
        moved += 4 * n * p
    if case["kind"] == "update":
        moved += 4 * m * s
    return dict(bytes=count * moved, flops=flops)


# ---- the same in 64 bits ---------------------------------------------------------

def _omp64(Y, D, s):
    """OMP of every signal in float64: indices (m, s) ascending, coefficients (m, s), and which of
    them count (a signal that is fitted exactly stops early: the start's atoms are signals)."""
    m = Y.shape[0]
    taken = torch.zeros(m, D.shape[0], dtype=torch.bool, device=Y.device)
    idx = torch.empty(m, 0, dtype=torch.int64, device=Y.device)
    on = torch.empty(m, 0, dtype=torch.bool, device=Y.device)
    r, yy = Y, Y.square().sum(1, keepdim=True)
    for _ in range(s):
        on = torch.cat([on, r.square().sum(1, keepdim=True) > 1e-6 * yy], 1)
        j = (r @ D.T).abs().masked_fill_(taken, -1.0).argmax(1, keepdim=True)
        taken.scatter_(1, j, True)
        idx = torch.cat([idx, j], 1)
        A = D[idx]
        x = torch.linalg.solve(A @ A.transpose(1, 2), A @ Y[:, :, None])
        r = Y - (A.transpose(1, 2) @ x)[:, :, 0]
    order = idx.argsort(1)
    on = on.gather(1, order)
    return idx.gather(1, order), x[:, :, 0].gather(1, order) * on, on


def _packed(x, on):
    """The coefficients that count, in order, in a buffer of m * s values."""
    out = torch.zeros(x.numel(), dtype=x.dtype, device=x.device)
    out[:int(on.sum())] = x[on]
    return out


def _update64(Y, D, idx, x):
    """The Jacobi atom update in float64: new atoms, new coefficients, RMSE before and after."""
    E = Y - torch.einsum("ms,msp->mp", x, D[idx])
    flat = idx.reshape(-1)
    U = torch.zeros_like(D).index_add_(0, flat, (x[:, :, None] * E[:, None, :]).reshape(-1, D.shape[1]))
    r = torch.zeros(D.shape[0], dtype=D.dtype, device=D.device).index_add_(0, flat, x.square().reshape(-1))
    V = U + r[:, None] * D
    norm = V.norm(dim=1, keepdim=True)
    N = torch.where(norm > 0, V / norm.clamp(min=1e-300), D)
    c = torch.where(norm[:, 0] > 0, (D * N).sum(1), torch.ones_like(r))
    xn = torch.einsum("mp,msp->ms", E, N[idx]) + c[idx] * x
    after = Y - torch.einsum("ms,msp->mp", xn, N[idx])
    yy = Y.square().sum()
    return N, xn, [float((E.square().sum() / yy).sqrt()), float((after.square().sum() / yy).sqrt())]


def _train64(case, seed):
    """Mean loss of the pass and the last batch's gradients, in float64."""
    Y, sup, weights = _train_inputs(case, seed)
    losses = []
    for r0 in range(0, case["m"] - case["batch"] + 1, case["batch"]):
        w = [torch.from_numpy(np.asarray(a, np.float32)).cuda().double().requires_grad_() for a in weights]
        y, at = Y[r0:r0 + case["batch"]].double(), sup[r0:r0 + case["batch"]].long()
        a = torch.nn.functional.gelu(y @ w[0].T + w[1])
        a = torch.nn.functional.gelu(a @ w[2].T + w[3])
        z = a @ w[4].T + w[5]
        t = torch.zeros_like(z).scatter_(1, at, 1.0)
        loss = torch.nn.functional.binary_cross_entropy_with_logits(z, t, reduction="sum") / case["batch"]
        losses.append(float(loss.detach()))
    return dict(loss=sum(losses) / len(losses), grad=[g.contiguous() for g in torch.autograd.grad(loss, w)])


def exact(case, seed):
    kind, s = case["kind"], case["s"]
    if kind == "train":
        return _train64(case, seed)
    Y, D = _inputs(case, seed)
    atoms, coefficients = [], []
    for k in range(Y.shape[0]):
        y, d = Y[k].double(), D[k].double()
        if kind == "update":
            idx, x = _given_x(Y[k], D[k], s)
            x, on = x.double(), torch.ones_like(idx, dtype=torch.bool)
        else:
            parts = [_omp64(part, d, s) for part in y.split(20000)]
            idx, x, on = (torch.cat([q[k] for q in parts]) for k in range(3))
        if kind == "encode":
            return dict(colptr=None, rowidx=None, val=_packed(x, on))
        new, xn, rmse = _update64(y, d, idx, x)
        atoms.append(new)
        coefficients.append(_packed(xn, on))
    out = dict(D=torch.stack(atoms), colptr=None, rowidx=None, val=torch.stack(coefficients))
    if kind != "batch":
        out.update(D=atoms[0], val=coefficients[0])
    if case.get("precision", "fp32") != "fp32":
        out["val"] = None  # other atoms are chosen for some signals, as they should be
    if case.get("track"):
        out["rmse"] = rmse
    return out
