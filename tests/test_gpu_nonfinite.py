"""The FP32 form on samples whose sums or powers are not finite: infinities, NaNs and overflow where the FP32 sums of
melt_forward_components have them, in every bin (frames of one sort, of both, and side by side)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

INF, NAN = np.inf, np.nan


@pytest.mark.parametrize("name,values", [
    ("powers overflow", dict(scale=1e25)), ("sums overflow", dict(fill=3e38)), ("all infinite", dict(fill=INF)),
    ("all NaN", dict(fill=NAN)), ("sparse", dict(at={700: INF, 5000: NAN, 9000: -INF, 9003: INF, 9100: NAN, 20000: 1e30})),
    ("last sample", dict(at={-1: NAN, 12: -INF}))])
@pytest.mark.parametrize("n_fft,hop,n_mels,n_mfcc", [(400, 160, 80, 0), (404, 100, 13, 0), (200, 88, 100, 20)])
def test_masks(name, values, n_fft, hop, n_mels, n_mfcc):
    import torch

    import __graft_entry__
    __graft_entry__.build()
    from oracle import melt_oracle as O
    from paper_2606_01009_gb300 import melt
    kw = dict(sr=16000.0, n_fft=n_fft, hop=hop, n_mels=n_mels, precision="fp32")
    x = np.random.default_rng(n_fft).standard_normal(n_fft + hop * 300).astype(np.float32) * np.float32(values.get("scale", 1))
    if "fill" in values:
        x[:] = values["fill"]
    for k, v in values.get("at", {}).items():
        x[k] = v
    wave = torch.from_numpy(np.pad(x, (0, -len(x) % 4))).cuda()
    comp = melt.Frontend(**kw)
    T = comp.total_frames([len(x)])
    ri = torch.empty(T, 2 * n_mels, device="cuda")
    melt.melt_forward_components(comp.handle, wave, None, [len(x)], ri)
    R, I = ri[:, :n_mels], ri[:, n_mels:]
    want = torch.log(R * R + I * I + 1e-10)
    fe = melt.Frontend(n_mfcc=n_mfcc, **kw) if n_mfcc else comp
    got = fe(wave, None, [len(x)])
    fe.sync()
    if n_mfcc:  # NaN wherever a term is NaN or infinities of both signs meet
        D = torch.from_numpy(O.dct2_ortho(n_mfcc, n_mels)).cuda().float()
        assert torch.equal(torch.isfinite(got).all(1), torch.isfinite(want).all(1))
        want = want @ D.T
        ok = torch.isfinite(want)
        assert torch.equal(torch.isfinite(got)[ok], ok[ok])
        return
    assert torch.equal(torch.isnan(got), torch.isnan(want)), name
    assert torch.equal(torch.isposinf(got), torch.isposinf(want)), name
