"""A wait of the CTA-pair kernel that runs out: a child process on the checked build, one load left out (withheld_pair_load_case.py)."""
import os
import subprocess
import sys
from pathlib import Path

import pytest

pytestmark = pytest.mark.gpu
ROOT = Path(__file__).resolve().parent.parent


@pytest.mark.parametrize("load", [1, 2, 3, 4, 5])  # V, Q rows, dO rows, dO columns, Q columns
def test_both_ctas_unwind(load):
    import torch

    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    env = dict(os.environ, NSP_LIBRARY=str(ROOT / "paper_2609_22755_b200" / "libnsp_checked.so"))
    r = subprocess.run([sys.executable, str(ROOT / "tests" / "withheld_pair_load_case.py"), str(load)], env=env,
                       capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr
    code = int(r.stdout.split("status ")[1].split()[0])
    assert code == 5  # NSP_ERR_DEVICE_TIMEOUT
