"""FP8 layouts whose staging ring has an odd number of slots (3, 5 and 7; with the MFCC's DCT on the
tensor cores too), fewer than a tile's chunks or more, over many turns of the ring, against the same
rounded operands in FP64 within the tensor-core forms' accumulation allowance (helpers.acc_rel, dct_rel)."""
import numpy as np
import pytest

from oracle import melt_oracle as O
from tests.helpers import acc_rel, dct_rel, gpu_features, oracle_features, rounded_log_bound

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_fft,hop,n_mels,n_mfcc", [
    (400, 160, 80, 0), (400, 200, 128, 0), (512, 224, 100, 0), (640, 256, 80, 0), (640, 256, 128, 0),
    (1024, 128, 128, 0), (400, 160, 80, 40), (400, 200, 128, 40), (640, 256, 128, 40)])
def test_odd_rings(n_fft, hop, n_mels, n_mfcc):
    import __graft_entry__
    __graft_entry__.build()
    from paper_2606_01009_gb300 import melt
    kw = dict(sr=16000.0, n_fft=n_fft, hop=hop, n_mels=n_mels, fmin=0.0, fmax=8000.0)
    g = np.random.default_rng(n_fft + hop + n_mels)
    frames = [128 * 60 + 9] + [40] * 500  # three and more tile pairs to a cluster
    clips = [(g.standard_normal(n_fft + hop * (f - 1)) * 10.0 ** g.uniform(-3, 0)).astype(np.float32) for f in frames]
    spec = O.MelTSpec(**kw)
    got = gpu_features(melt.Frontend(precision="fp8", n_mfcc=n_mfcc, **kw), clips)
    ref, bound = oracle_features(spec, clips, rounded="fp8"), rounded_log_bound(spec, clips, "fp8", acc_rel("fp8", n_fft, hop))
    if n_mfcc:
        D = O.dct2_ortho(n_mfcc, n_mels)
        bound = bound @ np.abs(D).T + dct_rel("fp8", n_mels) * (np.abs(ref) @ np.abs(D).T)
        ref = ref @ D.T
    assert np.all(np.abs(got - ref) <= bound)
