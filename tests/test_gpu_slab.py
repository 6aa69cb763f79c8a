"""The FP32 form on the tensor cores (three-part split operands, K slabs): edges of
tiles, blocks, slabs and chunks, geometries with odd hops, and samples the
split cannot hold.  Tolerance: the worst-case bound of the FP32 sum that the
form has always been held to (helpers.log_error_bound with n + 2 roundings);
what the split drops, below 2^-24 of each product, is inside its "+ 2"."""
import numpy as np
import pytest

from oracle import melt_oracle as O
from tests.helpers import (U32, acc_rel, fp32_sum_error, gpu_features, log_error_bound, oracle_features,
                           rounded_log_bound)

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def melt():
    import torch
    assert torch.cuda.is_available()
    import __graft_entry__
    __graft_entry__.build()
    from paper_2606_01009_gb300 import melt as m
    return m


def _clips(n_fft, hop, frames, seed):
    g = np.random.default_rng(seed)
    return [(g.standard_normal(n_fft + hop * (f - 1) + g.integers(0, hop)) * 10.0 ** g.uniform(-3, 0)).astype(np.float32)
            for f in frames]


# (n_fft, hop): one K-step, hop = N, hops that leave 4, 8, 12 of a slab's 16
# columns, a short last slice, one slice, many slices in stages of four (the
# last one shorter), and the shortest hop of the longest frame
GEOM = [(16, 16), (64, 64), (400, 160), (400, 100), (404, 12), (200, 88), (1200, 160), (1024, 256), (400, 400),
        (400, 20), (480, 16), (4096, 1024), (4096, 4)]


@pytest.mark.parametrize("n_fft,hop", GEOM)
@pytest.mark.parametrize("n_mels", [1, 80])
def test_geometries(melt, n_fft, hop, n_mels):
    kw = dict(sr=16000.0, n_fft=n_fft, hop=hop, n_mels=n_mels, fmin=0.0, fmax=8000.0)
    spec = O.MelTSpec(**kw)
    clips = _clips(n_fft, hop, [1, 2, 127, 128, 129, 300], n_fft + hop)
    got = gpu_features(melt.Frontend(precision="fp32", **kw), clips)
    assert np.all(np.abs(got - oracle_features(spec, clips)) <= log_error_bound(spec, clips, fp32_sum_error(n_fft)))


@pytest.mark.parametrize("n_mels,n_mfcc", [(8, 0), (17, 0), (81, 0), (96, 96), (100, 0), (128, 0), (128, 128), (81, 13)])
@pytest.mark.parametrize("tiles", [1, 3, 200])
def test_blocks_and_batches(melt, n_mels, n_mfcc, tiles):
    """One and two blocks of bins, the wider splits of short batches, several units per cluster."""
    kw = dict(sr=16000.0, n_fft=64, hop=32, n_mels=n_mels, fmin=0.0, fmax=8000.0)
    clips = _clips(64, 32, [128 * tiles - 5], n_mels)
    got = gpu_features(melt.Frontend(precision="fp32", n_mfcc=n_mfcc, **kw), clips)
    spec = O.MelTSpec(**kw)
    ref, bound = oracle_features(spec, clips), log_error_bound(spec, clips, fp32_sum_error(64))
    if n_mfcc:
        D = O.dct2_ortho(n_mfcc, n_mels)
        bound = bound @ np.abs(D).T + (n_mels + 2) * U32 * (np.abs(ref) @ np.abs(D).T)
        ref = ref @ D.T
    assert np.all(np.abs(got - ref) <= bound)


def test_mfcc_without_eps(melt):
    """The padded bins' log of zero stays out of the DCT."""
    kw = dict(sr=16000.0, n_fft=64, hop=32, n_mels=81, fmin=0.0, fmax=8000.0, eps=0.0)
    clips = _clips(64, 32, [130], 5)
    got = gpu_features(melt.Frontend(precision="fp32", n_mfcc=13, **kw), clips)
    spec = O.MelTSpec(**kw)
    D = O.dct2_ortho(13, 81)
    ref, bound = oracle_features(spec, clips), log_error_bound(spec, clips, fp32_sum_error(64))
    bound = bound @ np.abs(D).T + (81 + 2) * U32 * (np.abs(ref) @ np.abs(D).T)
    assert np.isfinite(got).all() and np.all(np.abs(got - ref @ D.T) <= bound)


@pytest.mark.parametrize("value", [np.inf, -np.inf, np.nan, 3.0e38])
@pytest.mark.parametrize("n_fft,hop", [(400, 160), (400, 100)])
def test_values_the_split_cannot_hold(melt, value, n_fft, hop):
    """Only the frames that hold such a sample see it: inf where their power overflows, NaN where
    the FP32 sum is one (a zero basis value, or infinities of both signs), finite elsewhere."""
    kw = dict(sr=16000.0, n_fft=n_fft, hop=hop, n_mels=80, fmin=0.0, fmax=8000.0)
    spec = O.MelTSpec(**kw)
    clean = _clips(n_fft, hop, [200], 3)
    at = 70 * hop + 33
    dirty = [clean[0].copy()]
    dirty[0][at] = value
    got = gpu_features(melt.Frontend(precision="fp32", **kw), dirty)
    t = np.arange(got.shape[0])
    hit = (t * hop <= at) & (at < t * hop + n_fft)
    ref, bound = oracle_features(spec, clean), log_error_bound(spec, clean, fp32_sum_error(n_fft))
    assert np.all(np.abs(got - ref)[~hit] <= bound[~hit])
    for f in t[hit]:
        n = at - f * hop
        zero = (spec.Wr[:, n].astype(np.float32) == 0) | (spec.Wi[:, n].astype(np.float32) == 0)
        nan = np.isnan(value) | (np.isinf(value) & zero)
        assert np.array_equal(np.isnan(got[f]), np.broadcast_to(nan, got[f].shape))
        # |x w|^2 overflows FP32 for every other basis value that is not tiny
        big = ~zero & (np.maximum(np.abs(spec.Wr[:, n]), np.abs(spec.Wi[:, n])) > 1e-15)
        if not np.isnan(value):
            assert np.all(got[f][big & ~np.broadcast_to(nan, big.shape)] == np.inf)


@pytest.mark.parametrize("prec,n_fft,hop,n_mels,streamed", [
    ("bf16x3", 400, 160, 80, True), ("bf16x3", 400, 80, 81, True), ("bf16x3", 404, 48, 128, True),
    ("bf16x3", 1200, 160, 100, True), ("bf16", 1024, 256, 80, True), ("bf16", 1200, 160, 128, True),
    ("bf16x3", 640, 64, 40, False)])
@pytest.mark.parametrize("tiles", [1, 40])
def test_rounded_forms(melt, prec, n_fft, hop, n_mels, streamed, tiles):
    """Split BF16, and BF16 whose half basis is streamed (the slab kernel, or not where a tile has too
    many rows), against the same rounded operands in FP64, within the tensor-core forms'
    accumulation allowance (helpers.acc_rel), and against the single-CTA kernel."""
    kw = dict(sr=16000.0, n_fft=n_fft, hop=hop, n_mels=n_mels, fmin=0.0, fmax=8000.0)
    clips = _clips(n_fft, hop, [1, 128 * tiles + 3], n_fft + n_mels)
    spec = O.MelTSpec(**kw)
    fe = melt.Frontend(precision=prec, **kw)
    plan = melt.melt_plan_get(fe.handle)
    assert ((plan["cta_pair"], plan["basis_resident"]) == (1, 0)) == streamed
    got, ref = gpu_features(fe, clips), oracle_features(spec, clips, rounded=prec)
    assert np.all(np.abs(got - ref) <= rounded_log_bound(spec, clips, prec, acc_rel(prec, n_fft, hop)))
    single = dict(basis_resident=0, a_buffers=1, prefetch_tiles=2, basis_slots=2, ksteps_per_slot=1, cta_pair=0,
                  schedule=0)
    melt.melt_plan_set(fe.handle, single)
    np.testing.assert_array_equal(gpu_features(fe, clips), got)  # the single-CTA kernel's sums, bit for bit
