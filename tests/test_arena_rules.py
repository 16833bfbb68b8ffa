"""The memory destroyed plans leave to later ones (csrc/nsp_arena.cu): its rules, compiled for the host against a stand-in
for the CUDA runtime in which work finishes when the test says so."""
import subprocess
from pathlib import Path

import pytest

ROOT = Path(__file__).resolve().parent.parent
SCENARIOS = ["two_streams", "back_pressure", "order_behind_construction", "recycled_stream_address", "reuse_and_trim", "sizes"]


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    out = tmp_path_factory.mktemp("arena") / "arena_case"
    csrc = ROOT / "paper_2609_22755_b200" / "csrc"
    subprocess.run(["g++", "-std=c++17", "-Wall", "-pthread", "-I", str(ROOT / "tests" / "fake_cuda"), "-I", str(csrc), "-x", "c++",
                    str(csrc / "nsp_arena.cu"), str(ROOT / "tests" / "arena_case.cpp"), "-o", str(out)], check=True)
    return out


@pytest.mark.parametrize("scenario", SCENARIOS)
def test_arena(program, scenario):
    r = subprocess.run([str(program), scenario], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout + r.stderr
