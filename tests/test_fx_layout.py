"""The shared-memory layouts of the fixed-point PIPG and of the discretization
by column classes hold what their kernels index, and the latter's warp roles
cover every column (tests/fx_layout_probe.cu, compiled on the host)."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
SRC = os.path.join(ROOT, "paper_2404_18034_gb300", "csrc")


@pytest.mark.parametrize("defs", [[], ["-DPDG_MODEL_3DOF"],
                                  [f'-DPDG_MODEL_HEADER="{HERE}/models/pdg_model_vertical.cuh"']],
                         ids=["6dof", "3dof", "vertical"])
def test_layouts_hold_what_the_kernels_index(tmp_path, defs):
    nvcc = os.environ.get("NVCC", shutil.which("nvcc") or "nvcc")
    if not shutil.which(nvcc) and not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    exe = str(tmp_path / "fx_layout_probe")
    subprocess.check_call([nvcc, "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a", "-I", SRC,
                           "-I", os.path.join(ROOT, "include")] + defs +
                          [os.path.join(HERE, "fx_layout_probe.cu"), "-o", exe])
    r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and r.stdout.startswith("OK"), r.stdout
    assert int(r.stdout.split()[1]) > 500
