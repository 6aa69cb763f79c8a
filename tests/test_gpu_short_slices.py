"""Pair kernels at hops of one to seven K-steps a slice (the walk of the K-steps changes at three and at six), with whole
and short last slices: BF16 log-Mel against the single-CTA kernel's sums bit for bit, MFCC and FP8 against the
same rounded operands in FP64 within the tensor-core forms' allowances (helpers.acc_rel, dct_rel)."""
import numpy as np
import pytest

from oracle import melt_oracle as O
from tests.helpers import acc_rel, dct_rel, gpu_features, oracle_features, rounded_log_bound

pytestmark = pytest.mark.gpu


def _frontend(prec, n_fft, hop, n_mels, n_mfcc=0):
    import __graft_entry__
    __graft_entry__.build()
    from paper_2606_01009_gb300 import melt
    kw = dict(sr=16000.0, n_fft=n_fft, hop=hop, n_mels=n_mels, fmin=0.0, fmax=8000.0)
    g = np.random.default_rng(n_fft + hop)
    clips = [(g.standard_normal(n_fft + hop * (f - 1)) * 10.0 ** g.uniform(-3, 0)).astype(np.float32)
             for f in [1, 129, 128 * 40 + 3]]
    return melt, melt.Frontend(precision=prec, n_mfcc=n_mfcc, **kw), O.MelTSpec(**kw), clips


@pytest.mark.parametrize("n_fft,hop", [(16, 16), (256, 16), (248, 16), (256, 32), (300, 32), (400, 48), (404, 64), (400, 80),
                                       (388, 96), (400, 112)])
@pytest.mark.parametrize("n_mels", [13, 80])
def test_bf16(n_fft, hop, n_mels):
    melt, fe, spec, clips = _frontend("bf16", n_fft, hop, n_mels)
    plan = melt.melt_plan_get(fe.handle)
    assert (plan["cta_pair"], plan["basis_resident"]) == (1, 1)
    got = gpu_features(fe, clips)
    melt.melt_plan_set(fe.handle, dict(basis_resident=0, a_buffers=1, prefetch_tiles=2, basis_slots=2, ksteps_per_slot=1,
                                       cta_pair=0, schedule=0))
    np.testing.assert_array_equal(gpu_features(fe, clips), got)


@pytest.mark.parametrize("prec,n_fft,hop,n_mels,n_mfcc", [("bf16", 256, 16, 40, 13), ("bf16", 400, 48, 80, 40),
                                                          ("fp8", 256, 32, 40, 0), ("fp8", 400, 96, 80, 40),
                                                          ("fp8", 500, 160, 40, 0)])
def test_mfcc_and_fp8(prec, n_fft, hop, n_mels, n_mfcc):
    _, fe, spec, clips = _frontend(prec, n_fft, hop, n_mels, n_mfcc)
    got, ref = gpu_features(fe, clips), oracle_features(spec, clips, rounded=prec)
    bound = rounded_log_bound(spec, clips, prec, acc_rel(prec, n_fft, hop))
    if n_mfcc:
        D = O.dct2_ortho(n_mfcc, n_mels)
        bound = bound @ np.abs(D).T + dct_rel(prec, n_mels) * (np.abs(ref) @ np.abs(D).T)
        ref = ref @ D.T
    assert np.all(np.abs(got - ref) <= bound)
