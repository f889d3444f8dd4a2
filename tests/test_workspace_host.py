"""The list map's memory is optional: what an evaluation allocates after it is
not refused for it (the workspace against a played device memory, on the CPU)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_lists_give_way(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("no nvcc")
    exe = str(tmp_path / "workspace_host")
    subprocess.run([nvcc, "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a", "-I",
                    os.path.join(ROOT, "paper_2208_05683_gb300", "csrc"), "-o", exe,
                    os.path.join(ROOT, "tests", "workspace_host.cu")], check=True)
    p = subprocess.run([exe], capture_output=True, text=True)
    assert p.returncode == 0 and p.stdout.endswith("ok\n"), p.stdout
