"""The status record of a bounded wait that ran out says which wait it was."""
import os
import subprocess
import sys
from pathlib import Path

import pytest

pytestmark = pytest.mark.gpu
ROOT = Path(__file__).resolve().parent.parent


def test_record_of_a_missing_tile_names_the_load():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    env = dict(os.environ, NSP_LIBRARY=str(ROOT / "paper_2609_22755_b200" / "libnsp_checked.so"))
    r = subprocess.run([sys.executable, str(ROOT / "tests" / "withheld_load_case.py")], env=env, capture_output=True, text=True,
                       timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr
