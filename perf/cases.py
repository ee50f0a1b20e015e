"""Performance cases of the library: what a user's program has it do, through the
public entry points of ``paper_1411_2860_gb300``.

Four kinds of work:
  gemm   one projected product, ``proj_gemm`` (BF16, split BF16, E4M3 and FP64 components)
  train  forward and backward of the differentiable product, ``proj_matmul`` under autograd
  conv   one projected cross-correlation, ``proj_conv`` (Haar and DCT-II)
  batch  many uneven products and correlations in one ``BatchPlan``

Sizes are those of the benchmark's workloads (face matching, differentiated layer,
audio correlation, uneven batch, FP64 product) and smaller, larger and ragged ones
between them.
"""
import math

import numpy as np
import torch

import paper_1411_2860_gb300 as pj

DEV = "cuda"
MOST_MNK = 4096 * 10304 * 2048   # the largest single product
L_GEMM = 8                       # group size of every product here (the library's default)


def listed():
    return [
        # A short query against a small table: one tile or two, bound by latency and launches.
        dict(name="gemm-small", kind="gemm", M=64, N=96, K=512, dtype="f32", compute="bf16", split=1, lead=0,
             block=128, lp1=4),
        # The plain FP64 product of the precision sweep, exact (R = block).
        dict(name="gemm-fp64", kind="gemm", M=256, N=256, K=512, dtype="f64", compute="f64", split=1, lead=0,
             block=128, lp1=8),
        # An ordinary product whose rows no copy engine can address (odd pitches), most projections
        # kept, hi/lo components.
        dict(name="gemm-ragged", kind="gemm", M=1000, N=777, K=3001, dtype="f32", compute="bf16", split=2, lead=0,
             block=128, lp1=6),
        # Face matching, a quarter of the projections kept: throughput before precision.
        dict(name="face-r128", kind="gemm", M=4096, N=2048, K=10304, dtype="f32", compute="bf16", split=1, lead=0,
             block=512, lp1=2),
        # Face matching at the 1e-3 error point: every projection, lo terms on the first.
        dict(name="face-lead1", kind="gemm", M=4096, N=2048, K=10304, dtype="f32", compute="bf16", split=2, lead=1,
             block=512, lp1=8),
        # A smaller batch of probes through the FP8 components with block scales.
        dict(name="gemm-e4m3", kind="gemm", M=1500, N=2048, K=10304, dtype="f32", compute="e4m3", split=2, lead=0,
             block=512, lp1=8),
        # A training step of the differentiated layer, a quarter of the projections kept.
        dict(name="layer-step", kind="train", M=8192, N=4096, K=4096, dtype="bf16", block=256, lp1=2, saved=False),
        # A small layer with sizes that fill no tile, keeping the forward's projections for the backward.
        dict(name="layer-small", kind="train", M=1111, N=776, K=1000, dtype="bf16", block=128, lp1=2, saved=True),
        # Cover-song style matching: a long signal against 64 templates, exact (R = T).
        dict(name="conv-full", kind="conv", S=1 << 20, T=4096, nt=64, basis="haar", L=64, lp1=64),
        # The same search at 1/16 of the components: a coarse pass, bound by its output.
        dict(name="conv-r256", kind="conv", S=1 << 20, T=4096, nt=64, basis="haar", L=64, lp1=4),
        # A shorter ragged signal, 37 templates, the DCT basis at half the components.
        dict(name="conv-dct2", kind="conv", S=300001, T=2048, nt=37, basis="dct2", L=8, lp1=4),
        # Uneven products and correlations planned once and run as one launch sequence.
        dict(name="batch", kind="batch", gemms=40, convs=20, sizes=1, block=128, lp1=8, split=2),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["gemm", "gemm", "gemm", "gemm", "train", "train", "conv", "conv", "conv", "batch"])
    if kind == "gemm":
        if rng.random() < 0.15:
            return dict(kind="gemm", M=_log(rng, 24, 384), N=_log(rng, 24, 384), K=_log(rng, 64, 768), dtype="f64",
                        compute="f64", split=1, lead=0, block=128, lp1=rng.choice([1, 2, 4, 8]))
        while True:
            M, N, K = _log(rng, 32, 8192), _log(rng, 32, 4096), _log(rng, 64, 10304)
            if M * N * K <= MOST_MNK:
                break
        if rng.random() < 0.6:   # row pitches a copy engine can address; the rest as drawn
            N, K = -(-N // 8) * 8, -(-K // 8) * 8
        compute = "e4m3" if rng.random() < 0.2 else "bf16"
        lp1 = rng.choice([1, 2, 2, 3, 4, 4, 5, 6, 7, 8, 8, 8])
        split = rng.choice([1, 2])
        lead = rng.choice([0, 1, 2]) if compute == "bf16" and split == 2 and lp1 > 2 else 0
        return dict(kind="gemm", M=M, N=N, K=K, dtype=rng.choice(["f32", "f32", "bf16"]), compute=compute,
                    split=split, lead=lead, block=rng.choice([128, 256, 512]), lp1=lp1)
    if kind == "train":
        while True:
            M, N, K = _log(rng, 512, 8192), _log(rng, 256, 4096), _log(rng, 256, 4096)
            if M * N * K >= 1 << 27:
                break
        if rng.random() < 0.75:
            N, K = -(-N // 8) * 8, -(-K // 8) * 8
        return dict(kind="train", M=M, N=N, K=K, dtype=rng.choice(["bf16", "bf16", "f32"]),
                    block=rng.choice([128, 256]), lp1=rng.choice([1, 2, 2, 4, 8]), saved=rng.random() < 0.5)
    if kind == "conv":
        basis, L = rng.choice([("haar", 64), ("haar", 64), ("dct2", 8)])
        T = 64 * rng.choice([4, 8, 16, 24, 32, 48, 64])
        lp1 = rng.choice([p for p in ((1, 4, 16, 64) if basis == "haar" else (2, 4, 8)) if p * T // L % 64 == 0])
        return dict(kind="conv", S=max(_log(rng, 1 << 13, 1 << 20), 2 * T), T=T, nt=rng.randint(1, 64), basis=basis,
                    L=L, lp1=lp1)
    return dict(kind="batch", gemms=rng.randint(4, 40), convs=rng.randint(0, 20), sizes=rng.randint(2, 1 << 20),
                block=128, lp1=rng.choice([2, 4, 8, 8]), split=rng.choice([1, 2]))


# ----------------------------------------------------------------- inputs --

_DTYPE = {"f64": torch.float64, "f32": torch.float32, "bf16": torch.bfloat16}


def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _probes(M, K, g):
    """M smooth rows quantised to 256 grey levels in [0, 1]: rows of flattened images."""
    z = torch.randn((M, K), generator=g, device=DEV)
    f = torch.fft.rfftfreq(K, device=DEV)
    z = torch.fft.irfft(torch.fft.rfft(z) * torch.exp(-2.0 * (math.pi * 4.0 * f) ** 2), n=K)
    lo, hi = z.amin(dim=1, keepdim=True), z.amax(dim=1, keepdim=True)
    return torch.round(255.0 * (z - lo) / (hi - lo)) / 255.0


def _gemm_inputs(c, seed):
    g = _gen(seed)
    M, N, K = c["M"], c["N"], c["K"]
    if c["dtype"] == "f64":     # i.i.d. uniform [-1, 1)
        A = torch.rand((M, K), generator=g, device=DEV, dtype=torch.float64) * 2 - 1
        B = torch.rand((K, N), generator=g, device=DEV, dtype=torch.float64) * 2 - 1
    else:                       # image rows against random features of unit length
        A = _probes(M, K, g)
        B = torch.randn((K, N), generator=g, device=DEV) / math.sqrt(K)
    return A.to(_DTYPE[c["dtype"]]), B.to(_DTYPE[c["dtype"]])


def _train_inputs(c, seed):
    g = _gen(seed)
    M, N, K = c["M"], c["N"], c["K"]
    X = (0.02 * torch.randn((M, K), generator=g, device=DEV)).to(_DTYPE[c["dtype"]])
    W = (0.02 * torch.randn((K, N), generator=g, device=DEV)).to(_DTYPE[c["dtype"]])
    return X, W, torch.randn((M, N), generator=g, device=DEV)   # the product is FP32, and so its gradient


def _conv_inputs(c, seed):
    """32 tones of 50 to 8000 Hz at 44.1 kHz, noise at 20 dB; templates cut from the signal."""
    g = _gen(seed)
    S, T, nt = c["S"], c["T"], c["nt"]
    r = np.random.default_rng(seed)
    f, a, ph = r.uniform(50.0, 8000.0, 32), r.uniform(0.1, 1.0, 32), r.uniform(0.0, 2 * np.pi, 32)
    n = torch.arange(S, device=DEV, dtype=torch.float64)
    s = torch.zeros(S, device=DEV, dtype=torch.float32)
    for i in range(32):
        cycles = torch.frac(n * float(f[i] / 44100.0))
        s += float(a[i]) * torch.sin(cycles.float() * float(2 * np.pi) + float(ph[i]))
    s += torch.randn(S, generator=g, device=DEV) * float(np.sqrt(np.sum(a * a) / 2 / 100.0))
    off = torch.from_numpy(r.integers(0, S - T + 1, nt)).to(DEV)
    return s, s[off[:, None] + torch.arange(T, device=DEV)[None, :]].contiguous()


T_BATCH = 1024   # template length of the batch's correlations


def _batch_sizes(c):
    r = np.random.default_rng(c["sizes"])
    gemms = [(int(r.integers(64, 2049)), int(r.integers(64, 2049)), int(r.integers(256, 8193)))
             for _ in range(c["gemms"])]
    return gemms, [int(r.integers(1 << 14, (1 << 20) + 1)) for _ in range(c["convs"])]


def _batch_inputs(c, seed):
    g = _gen(seed)
    gemms, convs = _batch_sizes(c)
    normal = lambda *shape: torch.randn(shape, generator=g, device=DEV)  # noqa: E731
    return [(normal(M, K), normal(K, N)) for M, N, K in gemms], [(normal(S), normal(1, T_BATCH)) for S in convs]


def prepare(case, seed):
    c = case
    if c["kind"] == "gemm":
        A, B = _gemm_inputs(c, seed)
        kw = dict(compute=c["compute"], split=c["split"], split_lead=c["lead"])
        return dict(kind="gemm", A=A, B=B, block=c["block"], R=c["lp1"] * c["block"] // L_GEMM, kw=kw)
    if c["kind"] == "train":
        X, W, dY = _train_inputs(c, seed)
        return dict(kind="train", X=X.requires_grad_(), W=W.requires_grad_(), dY=dY, block=c["block"],
                    R=c["lp1"] * c["block"] // L_GEMM, saved=c["saved"])
    if c["kind"] == "conv":
        s, k = _conv_inputs(c, seed)
        return dict(kind="conv", s=s, k=k, R=c["lp1"] * c["T"] // c["L"], basis=c["basis"], L=c["L"])
    gemms, convs = _batch_inputs(c, seed)
    outs, descs = [], []
    for A, B in gemms:
        outs.append(torch.empty((A.shape[0], B.shape[1]), device=DEV))
        descs.append(pj.batch_gemm(A, B, outs[-1], c["block"], c["lp1"] * c["block"] // L_GEMM, split=c["split"]))
    for s, k in convs:
        outs.append(torch.empty((s.shape[0] - T_BATCH + 1, 1), device=DEV))
        descs.append(pj.batch_conv(s, k, outs[-1], T_BATCH, split=c["split"]))
    return dict(kind="batch", plan=pj.BatchPlan(descs), outs=outs)


def run(state):
    s = state
    if s["kind"] == "gemm":
        return pj.proj_gemm(s["A"], s["B"], s["block"], s["R"], **s["kw"])
    if s["kind"] == "train":
        Y = pj.proj_matmul(s["X"], s["W"], s["block"], s["R"], save_projections=s["saved"])
        dX, dW = torch.autograd.grad(Y, (s["X"], s["W"]), s["dY"])
        return Y.detach(), dX, dW
    if s["kind"] == "conv":
        return pj.proj_conv(s["s"], s["k"], s["R"], s["basis"], s["L"])
    s["plan"].run()
    return s["outs"]


# ------------------------------------------------- work and 64-bit results --

def work(case):
    """Inputs read once, outputs written once; the reduced products (hi*hi, hi*lo and lo*hi
    where the option asks for them) and the projection of each operand."""
    c = case
    if c["kind"] in ("gemm", "train"):
        M, N, K, lp1 = c["M"], c["N"], c["K"], c["lp1"]
        es = {"f64": 8, "f32": 4, "bf16": 2}[c["dtype"]]
        Kp = -(-K // L_GEMM) * lp1
        project = 2.0 * (M + N) * K * lp1
        if c["kind"] == "train":
            return {"bytes": 2 * es * (M * K + K * N) + 4 * 2 * M * N, "flops": 6.0 * M * N * Kp + 2 * project}
        share = (c["lead"] or lp1) / lp1 if c["split"] == 2 else 0.0
        return {"bytes": es * (M * K + K * N) + (8 if es == 8 else 4) * M * N,
                "flops": 2.0 * M * N * Kp * (1 + 2 * share) + project}
    if c["kind"] == "conv":
        lags, R = c["S"] - c["T"] + 1, c["lp1"] * c["T"] // c["L"]
        return {"bytes": 4 * (c["S"] + c["nt"] * c["T"] + lags * c["nt"]), "flops": 2.0 * lags * c["nt"] * R}
    gemms, convs = _batch_sizes(c)
    terms = 3 if c["split"] == 2 else 1
    nb = sum(4 * (M * K + K * N + M * N) for M, N, K in gemms) + sum(4 * (2 * S + 1) for S in convs)
    fl = sum(2.0 * M * N * -(-K // 8) * c["lp1"] * terms + 2.0 * (M + N) * K * c["lp1"] for M, N, K in gemms)
    return {"bytes": nb, "flops": fl + sum(2.0 * (S - T_BATCH + 1) * T_BATCH * terms for S in convs)}


def _projector(basis, L, lp1):
    """The L x L orthogonal projector on the first lp1 basis functions, FP64."""
    i = np.arange(L)
    if basis == "dct2":
        C = np.cos(np.pi / L * (i[:, None] + 0.5) * i[None, :])
        C /= np.linalg.norm(C, axis=0)
        P = C[:, :lp1] @ C[:, :lp1].T
    else:   # Haar with lp1 a power of two: the functions constant on runs of L / lp1 samples
        run_ = L // lp1
        P = (i[:, None] // run_ == i[None, :] // run_) / run_
    return torch.from_numpy(P).to(DEV, torch.float64)


def _project_last(x, P):
    """x with each group of L consecutive values of its last dimension projected (the last zero-extended)."""
    L, K = P.shape[0], x.shape[-1]
    G = -(-K // L)
    x = torch.nn.functional.pad(x.double(), (0, G * L - K))
    return (x.reshape(*x.shape[:-1], G, L) @ P).reshape(*x.shape[:-1], G * L)[..., :K]


def _correlate(s, k):
    """Valid cross-correlation of s with every row of k, by an FP64 FFT."""
    n = 1 << (s.shape[0] - 1).bit_length()
    lags = s.shape[0] - k.shape[1] + 1
    F = torch.fft.rfft(s.double(), n=n)
    return torch.stack([torch.fft.irfft(F * torch.fft.rfft(row, n=n).conj(), n=n)[:lags] for row in k], dim=1)


def exact(case, seed):
    c = case
    if c["kind"] == "gemm":
        A, B = _gemm_inputs(c, seed)
        return _project_last(A, _projector("dct2", L_GEMM, c["lp1"])) @ B.double()
    if c["kind"] == "train":
        X, W, dY = (t.double() for t in _train_inputs(c, seed))
        P = _projector("dct2", L_GEMM, c["lp1"])
        Xp = _project_last(X, P)
        return Xp @ W, _project_last(dY @ W.t(), P), Xp.t() @ dY
    if c["kind"] == "conv":
        s, k = _conv_inputs(c, seed)
        return _correlate(s, _project_last(k, _projector(c["basis"], c["L"], c["lp1"])))
    gemms, convs = _batch_inputs(c, seed)
    P = _projector("dct2", L_GEMM, c["lp1"])
    return [_project_last(A, P) @ B.double() for A, B in gemms] + [_correlate(s, k.double()) for s, k in convs]
