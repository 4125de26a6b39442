"""State that a context keeps between calls (host code; no GPU)."""
import os
import subprocess
from pathlib import Path

ROOT = Path(__file__).resolve().parents[1]


def test_a_context_remembers_kernel_attributes_of_its_own_device_only(tmp_path):
    """A call made with another device current raises that device's limits; the next one has to raise the context's own."""
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    exe = tmp_path / "own_device"
    subprocess.check_call([nvcc, "-gencode", "arch=compute_100a,code=sm_100a", "-std=c++17", "-I", str(ROOT / "include"), "-I",
                           str(ROOT / "paper_2408_00167_b200" / "csrc"), "-o", str(exe), str(ROOT / "tests" / "native" / "own_device.cu")])
    assert subprocess.run([str(exe)], timeout=60).returncode == 0
