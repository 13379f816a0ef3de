"""The host's packed instruction forms against the plain code, compiled and run on the CPU."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA = os.environ.get("CUDA_HOME", "/usr/local/cuda")


def test_packed_runs_match_the_plain_code(tmp_path):
    exe = str(tmp_path / "pack_check")
    subprocess.run(["g++", "-O1", "-std=c++17", "-I", os.path.join(ROOT, "include"),
                    "-I", os.path.join(ROOT, "paper_1211_6193_gb300", "csrc"), "-I", os.path.join(CUDA, "include"),
                    os.path.join(ROOT, "tests", "host", "pack_check.cpp"), "-o", exe], check=True)
    out = subprocess.run([exe], check=True, capture_output=True, text=True).stdout.split()
    assert out[0] == "ok" and int(out[1]) > 100_000 and int(out[2]) > 10_000, out
