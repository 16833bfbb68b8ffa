"""The host's counting of list positions for large plans (csrc/nsp_plan_bases.cpp) against the sums small plans take."""
import subprocess
from pathlib import Path

ROOT = Path(__file__).resolve().parent.parent


def test_counted_positions_equal_the_sums(tmp_path):
    csrc = ROOT / "paper_2609_22755_b200" / "csrc"
    out = tmp_path / "plan_bases_case"
    subprocess.run(["g++", "-std=c++17", "-O1", "-Wall", "-D_GLIBCXX_ASSERTIONS", "-I", str(csrc), str(csrc / "nsp_plan_bases.cpp"),
                    str(ROOT / "tests" / "plan_bases_case.cpp"), "-o", str(out)], check=True)
    r = subprocess.run([str(out)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout + r.stderr
