"""Plan files of earlier library versions: a line that was tuned when a basis had other kernels to choose from is
not taken for the present one's."""
import pytest

pytestmark = pytest.mark.gpu


def test_line_from_before_the_slab_kernel(tmp_path):
    import torch

    import __graft_entry__
    __graft_entry__.build()
    from paper_2606_01009_gb300 import melt
    lengths = [16000] * 4
    wave = torch.randn(sum(lengths), device="cuda")
    old, new = str(tmp_path / "old.txt"), str(tmp_path / "new.txt")

    def tune(path):
        fe = melt.Frontend(precision="bf16x3")
        assert (melt.melt_plan_get(fe.handle)["cta_pair"], melt.melt_plan_get(fe.handle)["basis_resident"]) == (1, 0)
        out = torch.empty((fe.total_frames(lengths), fe.n_out), device="cuda")
        res = melt.melt_autotune_file(fe.handle, wave, None, lengths, out, path, reps=1)
        fe.close()
        return res

    best, hit = tune(new)
    assert not hit
    assert tune(new) == (best, True)
    line = open(new).read()
    cls = line.split(" : ")[0].split()[-1]
    gpu = line.split()[1]
    with open(old, "w") as f:  # what a version without the slab kernel wrote: its fastest, a single-CTA layout
        f.write(f"melt-plan-v1 {gpu} 400 160 80 2 0 0 0 {cls} : 0 1 2 2 1 0 0\n")
    best, hit = tune(old)
    assert not hit and len(open(old).read().splitlines()) == 2
