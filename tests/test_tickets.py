"""The counters by which the ranges of a scoring unit wait for one another (csrc/tickets.h), on host threads: every call leaves
them at zero, also one in which a range gives up, so that no call depends on the one before it."""
import subprocess
from pathlib import Path

ROOT = Path(__file__).resolve().parents[1]


def test_counters_are_zero_after_every_call_also_when_a_range_gives_up(tmp_path):
    exe = tmp_path / "tickets_model"
    subprocess.check_call(["g++", "-O1", "-std=c++17", "-pthread", "-I", str(ROOT / "paper_2408_00167_b200" / "csrc"),
                           "-o", str(exe), str(ROOT / "tests" / "native" / "tickets_model.cpp")])
    out = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert out.returncode == 0, out.stdout
