"""The slab kernel's rings over many turns: batches that give every cluster eight or more tile pairs,
against the single-CTA kernel's sums bit for bit (the two forms add the same products in the same order)."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,n_fft,hop,n_mels", [
    ("bf16x3", 256, 32, 128), ("bf16x3", 272, 32, 100),  # two slabs a tile: the shortest ring
    # rings that are no multiple of the converter teams, with a last slice of few slabs
    ("bf16x3", 512, 160, 80), ("bf16x3", 1024, 240, 80), ("bf16x3", 400, 160, 80), ("bf16", 1000, 480, 80),
    ("bf16", 2048, 400, 128), ("bf16", 800, 384, 128), ("bf16", 1024, 256, 80), ("bf16x3", 404, 48, 128),
])
def test_many_units(prec, n_fft, hop, n_mels):
    import torch

    import __graft_entry__
    __graft_entry__.build()
    from paper_2606_01009_gb300 import melt
    fe = melt.Frontend(sr=16000.0, n_fft=n_fft, hop=hop, n_mels=n_mels, precision=prec)
    plan = melt.melt_plan_get(fe.handle)
    assert (plan["cta_pair"], plan["basis_resident"]) == (1, 0)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    frames = 128 * (8 * sms + 1) + 5
    g = torch.Generator(device="cuda").manual_seed(n_fft + hop)
    lengths = [n_fft + hop * (frames - 1), n_fft + hop * 700]
    wave = torch.randn(sum((n + 3) // 4 * 4 for n in lengths), generator=g, device="cuda")
    got = fe(wave, None, lengths)
    melt.melt_plan_set(fe.handle, dict(basis_resident=0, a_buffers=1, prefetch_tiles=2, basis_slots=2, ksteps_per_slot=1,
                                       cta_pair=0, schedule=0))
    ref = fe(wave, None, lengths)
    melt.melt_sync(fe.handle)
    assert torch.equal(got.view(torch.int32), ref.view(torch.int32))
