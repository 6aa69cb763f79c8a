"""Default layouts where two A buffers would leave tiny staging chunks, or the slab kernel two converter
teams: the default avoids them, and the layout that it avoids still runs when set, with the same bits."""
import numpy as np
import pytest

from tests.helpers import gpu_features

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,n_fft,hop,n_mels,n_mfcc,want,other", [
    ("bf16", 400, 320, 64, 0, dict(cta_pair=1, basis_resident=1, a_buffers=1), dict(a_buffers=2)),
    ("fp8", 1000, 240, 128, 40, dict(cta_pair=1, basis_resident=1, a_buffers=1), dict(a_buffers=2)),
    ("bf16", 400, 160, 80, 0, dict(cta_pair=1, basis_resident=1, a_buffers=2), dict(a_buffers=1)),
    ("bf16", 944, 656, 64, 0, dict(cta_pair=0, basis_resident=0), dict(a_buffers=1)),
])
def test_default_plan(prec, n_fft, hop, n_mels, n_mfcc, want, other):
    import __graft_entry__
    __graft_entry__.build()
    from paper_2606_01009_gb300 import melt
    fe = melt.Frontend(sr=16000.0, n_fft=n_fft, hop=hop, n_mels=n_mels, n_mfcc=n_mfcc, precision=prec)
    plan = melt.melt_plan_get(fe.handle)
    assert {k: plan[k] for k in want} == want
    g = np.random.default_rng(hop)
    clips = [g.standard_normal(n_fft + hop * f).astype(np.float32) for f in (0, 130, 1500)]
    got = gpu_features(fe, clips)
    melt.melt_plan_set(fe.handle, {**plan, **other})
    np.testing.assert_array_equal(gpu_features(fe, clips), got)
