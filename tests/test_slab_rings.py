"""The slab kernel's ring plans, checked on the host from the planner's own code
(tests/native/slab_rings.cu, compiled with nvcc for sm_103a; its main() runs on
the CPU and launches nothing)."""
import os
import subprocess

import pytest

from tests.test_mlp_tmem_layout import ROOT, _nvcc


def test_ring_plans(tmp_path):
    nvcc = _nvcc()
    if nvcc is None:
        pytest.skip("nvcc not found")
    exe = str(tmp_path / "slab_rings")
    cmd = [nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17", "-O1",
           os.path.join(ROOT, "tests", "native", "slab_rings.cu"), "-o", exe]
    for d in ("paper_2606_01009_gb300/csrc", "include"):
        cmd += ["-I", os.path.join(ROOT, d)]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    run = subprocess.run([exe], capture_output=True, text=True)
    assert run.returncode == 0, run.stdout[-2000:]
