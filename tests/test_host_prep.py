"""The host's preparation of programs, compiled and run on the CPU: the packed instruction forms against
the plain code, and the reachable words of the shared array against executed accesses."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA = os.environ.get("CUDA_HOME", "/usr/local/cuda")


def run_check(name, tmp_path):
    exe = str(tmp_path / name)
    subprocess.run(["g++", "-O1", "-std=c++17", "-I", os.path.join(ROOT, "include"),
                    "-I", os.path.join(ROOT, "paper_1211_6193_gb300", "csrc"), "-I", os.path.join(CUDA, "include"),
                    os.path.join(ROOT, "tests", "host", name + ".cpp"), "-o", exe], check=True)
    p = subprocess.run([exe], capture_output=True, text=True)
    assert p.returncode == 0, p.stdout
    word, *counts = p.stdout.split()
    assert word == "ok", p.stdout
    return [int(c) for c in counts]


def test_packed_runs_match_the_plain_code(tmp_path):
    instrs, chained = run_check("pack_check", tmp_path)
    assert instrs > 100_000 and chained > 10_000


def test_shared_reach_covers_every_access(tmp_path):
    accesses, below = run_check("reach_check", tmp_path)
    assert accesses > 20_000 and below > 300


def test_shared_reach_is_analysed_once_for_alike_launches(tmp_path):
    launches, analyses = run_check("reach_memo_check", tmp_path)
    assert launches == 48_000 and analyses == 1
