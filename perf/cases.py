"""The work that is timed: MelT forwards of every operand form, the grouped and
host-buffer calls, the fused correction and its training step, each through the
public entry points of the Python binding.

Audio is drawn on the GPU from the seed: pink noise with amplitude-modulated
harmonic and chirp bursts, the kind of signal the repository's own workloads
hold, at a level per clip.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2606_01009_gb300 import melt

DEV = "cuda"
# (sr, n_fft, hop) of the repository's configurations
G16 = {"sr": 16000.0, "n_fft": 400, "hop": 160}
G22 = {"sr": 22050.0, "n_fft": 1024, "hop": 256}
CEP = {"sr": 16000.0, "n_fft": 1200, "hop": 160}
MAX_FLOPS = 64 * 2998 * 128000.0  # projection of the 64 x 30 s batch at 400/160/80


def _forward(**kw):
    c = {"kind": "forward", "precision": "bf16", "clips": 64, "samples": 480000, "n_mels": 80, "n_mfcc": 0,
         "fmin": 0.0, "fmax": 8000.0, "window": 0, "center": False, "input_ready": False, "level_lo": 0.0,
         "uneven": False, **G16}
    c.update(kw)
    return c


def listed():
    return [
        # one short utterance, alone: a streaming or interactive caller, where the launch is what counts
        _forward(name="utterance_1x4s_bf16", clips=1, samples=64000),
        # the default form on eight one-second clips: a small batch of commands
        _forward(name="commands_8x1s_fp32", precision="fp32", clips=8, samples=16000),
        # the headline batch: 64 segments of 30 s, audio already on the device, launches back to back
        _forward(name="batch_64x30s_bf16", input_ready=True),
        # the same batch in the default FP32 form
        _forward(name="batch_64x30s_fp32", precision="fp32"),
        # split BF16, for callers that want near-FP32 features: clips of 10 s at levels of -60..0 dBFS
        _forward(name="levels_256x10s_bf16x3", precision="bf16x3", clips=256, samples=160000, level_lo=-60.0),
        # e4m3 operands: the cheapest form's batch
        _forward(name="batch_64x30s_fp8", precision="fp8", input_ready=True),
        # MFCCs (DCT-II fused) of the headline batch
        _forward(name="mfcc40_64x30s_bf16", n_mfcc=40, input_ready=True),
        # one long recording through the long-window cepstral configuration, FP32
        _forward(name="cepstral_1x160s_fp32", precision="fp32", clips=1, samples=2560000, n_mels=128, n_mfcc=40,
                 window=1, **{k: v for k, v in CEP.items()}),
        # uneven clips of two frame geometries in one grouped call: a mixed training set
        {"name": "grouped_4096_bf16", "kind": "grouped", "precision": "bf16", "clips": 4096, "lo_s": 0.5, "hi_s": 30.0,
         "n_mels": 80},
        # features from host memory to host memory (the copies are part of the call)
        {"name": "host_64x30s_bf16", "kind": "host", "precision": "bf16", "clips": 64, "samples": 480000, "n_mels": 80,
         "level_lo": 0.0, **G16},
        # the learned correction applied while the features are made
        {"name": "correction_64x30s_bf16", "kind": "correction", "precision": "bf16", "clips": 64, "samples": 480000,
         "n_mels": 80, "hidden": 256, **G16},
        # one step of the correction's training: gradient of a gathered batch, then AdamW
        {"name": "train_step_1024", "kind": "train", "rows": 200000, "batch": 1024, "n_mels": 80, "hidden": 256},
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["forward"] * 6 + ["grouped", "host", "correction", "train"])
    if kind == "train":
        return {"kind": "train", "rows": _logint(rng, 5000, 200000), "batch": _logint(rng, 64, 4096),
                "n_mels": rng.choice([40, 64, 80, 128]), "hidden": rng.choice([64, 128, 256, 512])}
    if kind == "grouped":
        return {"kind": "grouped", "precision": rng.choice(["bf16", "bf16x3", "fp32"]), "clips": _logint(rng, 8, 1024),
                "lo_s": 0.5, "hi_s": rng.uniform(4.0, 30.0), "n_mels": rng.choice([40, 80, 128])}
    if kind == "correction":
        return {"kind": "correction", "precision": rng.choice(["bf16", "bf16", "fp32"]), "clips": _logint(rng, 1, 64),
                "samples": _logint(rng, 8000, 480000), "n_mels": rng.choice([40, 64, 80, 128]),
                "hidden": rng.choice([64, 128, 256]), **G16}
    if kind == "host":
        return {"kind": "host", "precision": rng.choice(["bf16", "fp32", "bf16x3", "fp8"]), "clips": _logint(rng, 1, 64),
                "samples": _logint(rng, 8000, 480000), "n_mels": 80, "level_lo": rng.choice([0.0, -60.0]), **G16}
    precision = rng.choice(["fp32", "fp32", "bf16", "bf16", "bf16x3", "fp8"])
    geom = rng.choice([G16, G16, G16, G22, CEP]) if precision != "fp8" else G16
    wide = precision in ("bf16", "bf16x3") and rng.random() < 0.2
    n_mels = rng.randrange(129, 513) if wide else rng.choice([13, 40, 64, 80, 80, 100, 128])
    n_mfcc = min(n_mels, rng.choice([13, 20, 40])) if not wide and rng.random() < 0.25 else 0
    samples = _logint(rng, 8000, 2560000)
    frames = max(1, samples // geom["hop"])
    most = MAX_FLOPS / (4.0 * geom["n_fft"] * n_mels * frames)
    clips = max(1, min(_logint(rng, 1, 1024), int(most)))
    paper = rng.random() < 0.3
    return _forward(precision=precision, clips=clips, samples=samples, n_mels=n_mels, n_mfcc=n_mfcc,
                    fmin=80.0 if paper else 0.0, fmax=7600.0 if paper else 8000.0, window=1 if paper else 0,
                    center=rng.random() < 0.2, input_ready=rng.random() < 0.3, level_lo=rng.choice([0.0, -60.0]),
                    uneven=rng.random() < 0.4, **geom)


# ------------------------------------------------------------------- inputs
def _pool(gen, sr, seconds=30.0, n=8):
    """n signals of `seconds` at `sr`, peak 1: pink noise and bursts of harmonic stacks and chirps."""
    L = int(seconds * sr)
    nfft = 1 << (L - 1).bit_length()
    spec = torch.randn(n, nfft // 2 + 1, generator=gen, device=DEV, dtype=torch.complex64)
    spec /= torch.arange(nfft // 2 + 1, device=DEV).clamp(min=1).sqrt()
    spec[:, 0] = 0
    x = torch.fft.irfft(spec, nfft)[:, :L]
    x = x / x.square().mean(1, keepdim=True).sqrt() * 0.03
    t = torch.arange(L, device=DEV, dtype=torch.float32) / sr
    u = lambda *s: torch.rand(*s, generator=gen, device=DEV)  # noqa: E731
    for b in range(24):
        start, length = u(n, 1) * (seconds - 0.8), 0.08 + 0.72 * u(n, 1)
        s = ((t[None] - start) / length).clamp(0, 1)
        env = (0.2 + 0.8 * u(n, 1)) * torch.sin(math.pi * s).square()
        if b % 2:
            f0, f1 = 50.0 * 150.0 ** u(n, 1), 50.0 * 150.0 ** u(n, 1)
            y = torch.sin(2 * math.pi * length * (f0 * s + 0.5 * (f1 - f0) * s * s))
        else:
            ph = 2 * math.pi * (80.0 + 320.0 * u(n, 1)) * length * s
            y = sum(torch.sin(h * ph) / h for h in (1, 2, 3, 5, 8, 13, 18))
        x += env * y
    return x / x.abs().amax(1, keepdim=True)


def _audio(case, gen, lengths, sr, pool=None):
    """Clips of the given lengths, packed at 4-float alignment: cut from the pool (looped), at a level per clip."""
    pool = _pool(gen, sr) if pool is None else pool
    n, P = pool.shape
    sizes = (lengths + 3) // 4 * 4
    offsets = np.concatenate([[0], np.cumsum(sizes)[:-1]]).astype(np.int64)
    wave = torch.zeros(int(sizes.sum()), device=DEV)
    g = np.random.Generator(np.random.PCG64(gen.initial_seed()))
    at = g.integers(0, P, len(lengths))
    lev = 10.0 ** (g.uniform(case.get("level_lo", 0.0), 0.0, len(lengths)) / 20.0)
    for b, (o, L) in enumerate(zip(offsets.tolist(), lengths.tolist())):
        src, s, done = pool[b % n], int(at[b]), 0
        while done < L:
            k = min(L - done, P - s)
            torch.mul(src[s:s + k], float(lev[b]), out=wave[o + done:o + done + k])
            done, s = done + k, 0
    return wave, offsets


def _lengths(case):
    L = np.full(case["clips"], case["samples"], dtype=np.int64)
    if case.get("uneven"):
        g = np.random.Generator(np.random.PCG64(case["clips"]))
        L = np.maximum(case["n_fft"], (L * g.uniform(0.3, 1.0, len(L))).astype(np.int64))
    return L


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _params(case, seed):
    """Xavier-uniform weights and small biases, packed; per-band statistics of log-Mel features."""
    M, Hd = case["n_mels"], case["hidden"]
    g = np.random.Generator(np.random.PCG64(seed))
    a = math.sqrt(6.0 / (M + Hd))
    W1, W2 = g.uniform(-a, a, (Hd, M)), g.uniform(-a, a, (M, Hd))
    p = melt.pack_mlp_params(W1, g.uniform(-0.1, 0.1, Hd), W2, g.uniform(-0.1, 0.1, M))
    return p, (-4.0 + 0.05 * np.arange(M)).astype(np.float32), g.uniform(2.0, 4.0, M).astype(np.float32)


class _State:
    """What a caller's program holds between calls; closes the library's handles with it."""

    def __init__(self, **kw):
        self.__dict__.update(kw)

    def __del__(self):
        torch.cuda.synchronize()
        if getattr(self, "group", None) is not None:
            self.group.close()
        for fe in getattr(self, "fes", []):
            fe.close()
        if getattr(self, "mlp", None) is not None:
            melt.melt_mlp_destroy(self.mlp)


def _frontend(case, geom=None, **kw):
    geom = geom or case
    return melt.Frontend(sr=geom["sr"], n_fft=geom["n_fft"], hop=geom["hop"], n_mels=case["n_mels"],
                         precision=case["precision"], **kw)


def _group_of(case):
    g = np.random.Generator(np.random.PCG64(case["clips"]))
    ids = (np.arange(case["clips"]) % 2).astype(np.int32)
    d = np.exp(g.uniform(math.log(case["lo_s"]), math.log(case["hi_s"]), case["clips"]))
    return ids, np.round(d * np.where(ids == 0, G16["sr"], G22["sr"])).astype(np.int64)


def prepare(case, seed):
    kind, gen = case["kind"], _gen(seed)
    if kind == "train":
        M = case["n_mels"]
        p, mu, sd = _params(case, seed)
        X = torch.randn(case["rows"], M, generator=gen, device=DEV) * torch.from_numpy(sd).to(DEV)
        X += torch.from_numpy(mu).to(DEV)
        T = X + 0.5 * torch.randn(case["rows"], M, generator=gen, device=DEV) + 1.0
        rows = torch.randperm(case["rows"], generator=gen, device=DEV)[:case["batch"]].contiguous()
        return _State(kind=kind, mlp=melt.melt_mlp_create(M, case["hidden"], p, mu, sd), X=X, T=T, rows=rows,
                      batch=int(rows.numel()), grads=torch.empty(p.size, device=DEV), loss=torch.zeros(1, device=DEV))
    if kind == "grouped":
        ids, lengths = _group_of(case)
        fes = [_frontend(case, G16, fmax=8000.0), _frontend(case, G22, fmax=8000.0)]
        wave, offsets = _audio(case, gen, lengths, G16["sr"])
        group = melt.GroupedFrontend(fes)
        out = torch.empty(group.total_frames(lengths, ids), case["n_mels"], device=DEV)
        return _State(kind=kind, fes=fes, group=group, wave=wave, offsets=offsets, lengths=lengths, ids=ids, out=out)
    lengths = _lengths(case)
    wave, offsets = _audio(case, gen, lengths, case["sr"])
    if kind == "forward":
        fe = _frontend(case, n_mfcc=case["n_mfcc"], fmin=case["fmin"], fmax=case["fmax"], window=case["window"],
                       center=case["center"])
    else:
        fe = _frontend(case)
    out = torch.empty(fe.total_frames(lengths), fe.n_out, device=DEV)
    st = _State(kind=kind, fes=[fe], fe=fe, wave=wave, offsets=offsets, lengths=lengths, out=out,
                ready=case.get("input_ready", False))
    if kind == "host":
        st.wave, st.out = wave.cpu().pin_memory(), torch.empty(out.shape, pin_memory=True)
    if kind == "correction":
        p, mu, sd = _params(case, seed)
        st.mlp = melt.melt_mlp_create(case["n_mels"], case["hidden"], p, mu, sd)
        melt.melt_basis_set_correction(fe.handle, st.mlp)
    return st


def run(st):
    if st.kind == "train":
        st.loss.zero_()
        melt.melt_mlp_grad(st.mlp, st.X, st.T, st.rows, st.batch, st.grads, st.loss)
        melt.melt_mlp_adamw_apply(st.mlp, st.grads)
        return {"grads": st.grads, "loss": st.loss}
    if st.kind == "grouped":
        return st.group(st.wave, st.offsets, st.lengths, st.ids, out=st.out)
    if st.kind == "host":
        melt.melt_forward_host(st.fe.handle, st.wave, st.offsets, st.lengths, st.out)
        return st.out
    return st.fe(st.wave, st.offsets, st.lengths, out=st.out, input_ready=st.ready)


# --------------------------------------------------------------------- work
def _frames(L, geom, center=False):
    L = L + (2 * (geom["n_fft"] // 2) if center else 0)
    return np.where(L < geom["n_fft"], 0, (L - geom["n_fft"]) // geom["hop"] + 1)


def work(case):
    M = case["n_mels"]
    if case["kind"] == "train":
        B, Hd = min(case["batch"], case["rows"]), case["hidden"]
        P = 2 * M * Hd + M + Hd
        # batch rows of X and T, parameters and both moments in and out, gradients out; five GEMMs of 2 B M Hd
        return {"bytes": 4.0 * (2 * B * M + 7 * P), "flops": 10.0 * B * M * Hd}
    if case["kind"] == "grouped":
        ids, L = _group_of(case)
        b = f = 0.0
        for g, geom in enumerate((G16, G22)):
            T = float(_frames(L[ids == g], geom).sum())
            b += 4.0 * float(L[ids == g].sum()) + 4.0 * T * M
            f += 4.0 * T * geom["n_fft"] * M
        return {"bytes": b, "flops": f}
    L = _lengths(case)
    T = float(_frames(L, case, case.get("center", False)).sum())
    n_out = case.get("n_mfcc", 0) or M
    flops = T * (4.0 * case["n_fft"] * M + 2.0 * M * case.get("n_mfcc", 0))
    if case["kind"] == "correction":
        flops += 4.0 * T * M * case["hidden"]
    return {"bytes": 4.0 * float(L.sum()) + 4.0 * T * n_out, "flops": flops}


# ------------------------------------------------------------- 64-bit values
def _basis64(case, geom):
    """[2M, N] window-folded cos / sin rows at the M interior Mel-spaced frequencies."""
    M, N = case["n_mels"], geom["n_fft"]
    mel = lambda f: 2595.0 * math.log10(1.0 + f / 700.0)  # noqa: E731
    lo, hi = mel(case.get("fmin", 0.0)), mel(case.get("fmax", 8000.0))
    f = 700.0 * (10.0 ** ((lo + (hi - lo) * torch.arange(1, M + 1, dtype=torch.float64) / (M + 1)) / 2595.0) - 1.0)
    n = torch.arange(N, dtype=torch.float64)
    w = 0.5 - 0.5 * torch.cos(2 * math.pi * n / (N - 1 if case.get("window", 0) else N))
    th = 2 * math.pi * f[:, None] * n[None] / geom["sr"]
    return torch.cat([w * torch.cos(th), w * torch.sin(th)]).to(DEV)


def _e4m3_rows(x, hop):
    """The FP8 form's operand: rows of `hop` samples, each rounded to e4m3 with the least power-of-two scale."""
    r = torch.nn.functional.pad(x, (0, -len(x) % hop)).view(-1, hop).double()
    a = r.abs().amax(1, keepdim=True)
    s = torch.where(a > 0, 2.0 ** torch.ceil(torch.log2((a / 448.0).clamp(min=1e-38))), torch.ones_like(a))
    return ((r / s).float().to(torch.float8_e4m3fn).double() * s).view(-1)[:len(x)]


def _logmel64(case, geom, x, W, D):
    """Log-Mel (or MFCC) rows of one clip in 64 bits."""
    if case.get("center"):
        p = geom["n_fft"] // 2
        x = torch.nn.functional.pad(x[None, None], (p, p), mode="reflect")[0, 0]
    x = _e4m3_rows(x, geom["hop"]) if case["precision"] == "fp8" else x.double()
    if len(x) < geom["n_fft"]:
        return torch.empty(0, len(W) // 2 if D is None else len(D), device=DEV, dtype=torch.float64)
    M, rows = len(W) // 2, []
    for part in x.unfold(0, geom["n_fft"], geom["hop"]).split(32768):
        p = part @ W.T
        v = torch.log(p[:, :M].square() + p[:, M:].square() + 1e-10)
        rows.append(v if D is None else v @ D.T)
    return torch.cat(rows)


def _mlp64(case, p, mu, sd, x):
    t = lambda a: torch.from_numpy(np.asarray(a)).to(DEV).double()  # noqa: E731
    W1, b1, W2, b2 = (t(a) for a in melt.unpack_mlp_params(p, case["n_mels"], case["hidden"]))
    xh = (x - t(mu)) / t(sd)
    return torch.cat([xc + torch.nn.functional.gelu(h @ W1.T + b1) @ W2.T + b2
                      for xc, h in zip(x.split(65536), xh.split(65536))])


def _train64(case, seed):
    st = prepare(case, seed)
    p, mu, sd = _params(case, seed)
    t = lambda a: torch.from_numpy(np.asarray(a)).to(DEV).double()  # noqa: E731
    prm = [t(a).requires_grad_() for a in melt.unpack_mlp_params(p, case["n_mels"], case["hidden"])]
    x, y = st.X[st.rows].double(), st.T[st.rows].double()
    out = x + torch.nn.functional.gelu((x - t(mu)) / t(sd) @ prm[0].T + prm[1]) @ prm[2].T + prm[3]
    se = (out - y).square().sum()
    g = torch.autograd.grad(se / out.numel(), prm)
    return {"grads": torch.cat([a.reshape(-1) for a in g]), "loss": se.detach().reshape(1)}


def exact(case, seed):
    if case["kind"] == "train":
        return _train64(case, seed)
    gen = _gen(seed)
    if case["kind"] == "grouped":
        ids, lengths = _group_of(case)
        geoms, sr = [(G16, G22)[g] for g in ids], G16["sr"]
    else:
        lengths = _lengths(case)
        geoms, sr = [case] * len(lengths), case["sr"]
    wave, offsets = _audio(case, gen, lengths, sr)
    D = None
    if case.get("n_mfcc"):
        M = case["n_mels"]
        k = torch.arange(case["n_mfcc"], dtype=torch.float64)[:, None]
        D = torch.cos(math.pi * k * (2 * torch.arange(M, dtype=torch.float64) + 1) / (2 * M)) * math.sqrt(2.0 / M)
        D[0] *= math.sqrt(0.5)
        D = D.to(DEV)
    W = {id(g): _basis64(case, g) for g in geoms}
    if case["precision"] == "fp8":
        W = {k: (w * 256.0).float().to(torch.float8_e4m3fn).double() / 256.0 for k, w in W.items()}
    out = torch.cat([_logmel64(case, g, wave[o:o + L], W[id(g)], D)
                     for g, o, L in zip(geoms, offsets.tolist(), lengths.tolist())])
    if case["kind"] == "correction":
        out = _mlp64(case, *_params(case, seed), out)
    return out
