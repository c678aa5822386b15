"""What must hold for the launch plans of every batch size, checked on the host (tests/plans.cu)."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
NVCC = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")


def test_no_two_ctas_with_tensor_memory_share_an_sm(tmp_path):
    """Batches 1 to 1024, CTA pairs by the cost model, never and always."""
    if not shutil.which(NVCC):
        pytest.skip("no nvcc")
    exe = str(tmp_path / "plans")
    subprocess.check_call([NVCC, "-gencode", "arch=compute_100a,code=sm_100a", "-O1", "-std=c++17", "-o", exe, os.path.join(HERE, "plans.cu")])
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout[:2000]
