"""FP8 converters: warp groups that take the staged chunks of a tile in turn.  Every count of quads a
lane holds (hops up to 256, whole and not), chunk counts that are odd and even, clips that end inside
a chunk and enough tiles that the turns cross from one tile to the next, against the same rounded
operands in FP64 within the tensor-core forms' accumulation allowance (helpers.acc_rel)."""
import numpy as np
import pytest

from oracle import melt_oracle as O
from tests.helpers import acc_rel, gpu_features, oracle_features, rounded_log_bound

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_fft,hop,n_mels", [(256, 32, 40), (400, 100, 80), (400, 160, 80), (512, 224, 64), (640, 256, 40)])
def test_fp8_chunks(n_fft, hop, n_mels):
    import __graft_entry__
    __graft_entry__.build()
    from paper_2606_01009_gb300 import melt
    kw = dict(sr=16000.0, n_fft=n_fft, hop=hop, n_mels=n_mels, fmin=0.0, fmax=8000.0)
    g = np.random.default_rng(n_fft + hop)
    frames = [1, 31, 128, 129, 300] + [33] * 180  # more pairs than clusters
    clips = [(g.standard_normal(n_fft + hop * (f - 1) + g.integers(0, hop)) * 10.0 ** g.uniform(-3, 0)).astype(np.float32)
             for f in frames]
    spec = O.MelTSpec(**kw)
    got = gpu_features(melt.Frontend(precision="fp8", **kw), clips)
    ref = oracle_features(spec, clips, rounded="fp8")
    assert np.all(np.abs(got - ref) <= rounded_log_bound(spec, clips, "fp8", acc_rel("fp8", n_fft, hop)))
