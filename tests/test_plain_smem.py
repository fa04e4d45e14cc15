"""The plain form's launches ask for shared memory that holds the layout of
each of their kernels (tests/plain_smem_probe.cu, compiled on the host): PIPG
form 3 on short grids runs fewer threads than the discretization, whose stage
buffers then need more than PIPG's layout has."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = os.path.join(ROOT, "paper_2404_18034_gb300", "csrc")


@pytest.mark.parametrize("defs", [[], ["-DPDG_MODEL_3DOF"]], ids=["6dof", "3dof"])
def test_plain_launches_hold_every_layout(tmp_path, defs):
    nvcc = os.environ.get("NVCC", shutil.which("nvcc") or "nvcc")
    if not shutil.which(nvcc) and not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    exe = str(tmp_path / "plain_smem_probe")
    subprocess.check_call([nvcc, "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a", "-I", SRC,
                           "-I", os.path.join(ROOT, "include")] + defs +
                          [os.path.join(ROOT, "tests", "plain_smem_probe.cu"), "-o", exe])
    r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and r.stdout.startswith("OK"), r.stdout
    assert int(r.stdout.split()[2]) > 0  # grids where PIPG's own layout is too small
    host = open(os.path.join(SRC, "pdg_mc.cu")).read()
    assert host.count("plain_total(h->n_max, NU, pl.Tp, ") == 3  # solve, step and no-allocation entry points
