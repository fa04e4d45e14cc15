"""Models of every accepted size compile with the fixed-point PIPG, and their
states' order in its node vectors is sound (tests/fx_order_probe.cu, compiled
on the host)."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
SRC = os.path.join(ROOT, "paper_2404_18034_gb300", "csrc")
MODELS = os.path.join(HERE, "models")


@pytest.mark.parametrize("nx,split,defs", [
    (15, 1, []), (8, 1, ["-DPDG_MODEL_3DOF"]),
    (8, 0, [f'-DPDG_MODEL_HEADER="{MODELS}/pdg_model_3dof_drag.cuh"']),
    (3, 0, [f'-DPDG_MODEL_HEADER="{MODELS}/pdg_model_vertical.cuh"']),
    (2, 0, [f'-DPDG_MODEL_HEADER="{MODELS}/pdg_model_vertical.cuh"', "-DPDG_VERTICAL_NX=2"])],
    ids=["6dof", "3dof", "drag", "three", "two"])
def test_state_order(tmp_path, nx, split, defs):
    nvcc = os.environ.get("NVCC", shutil.which("nvcc") or "nvcc")
    if not shutil.which(nvcc) and not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    exe = str(tmp_path / "fx_order_probe")
    subprocess.check_call([nvcc, "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a", "-I", SRC,
                           "-I", os.path.join(ROOT, "include")] + defs +
                          [os.path.join(HERE, "fx_order_probe.cu"), "-o", exe])
    r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and r.stdout.split() == ["OK", str(nx), str(split)], r.stdout
