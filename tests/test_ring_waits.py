"""The shared-memory rings' waits, checked on the host from the planner's and the
kernels' own code (tests/native/slab_rings.cu, fp8_chunks.cu, compiled with nvcc
for sm_103a; their main() runs on the CPU and launches nothing)."""
import os
import subprocess

import pytest

from tests.test_mlp_tmem_layout import ROOT, _nvcc


@pytest.mark.parametrize("name", ["slab_rings", "fp8_chunks"])
def test_waits(tmp_path, name):
    nvcc = _nvcc()
    if nvcc is None:
        pytest.skip("nvcc not found")
    exe = str(tmp_path / name)
    cmd = [nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17", "-O1",
           os.path.join(ROOT, "tests", "native", name + ".cu"), "-o", exe]
    for d in ("paper_2606_01009_gb300/csrc", "include"):
        cmd += ["-I", os.path.join(ROOT, d)]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    run = subprocess.run([exe], capture_output=True, text=True)
    assert run.returncode == 0, run.stdout[-2000:]
