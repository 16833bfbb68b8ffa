"""A wait of the CTA-pair kernel that runs out: a child process on the checked build, one load left out
(withheld_pair_load_case.py). The record names the wait."""
import os
import subprocess
import sys
from pathlib import Path

import pytest

pytestmark = pytest.mark.gpu
ROOT = Path(__file__).resolve().parent.parent


LOAD_KV, LOAD_Q, S_FULL, DQ_FULL, LD_FULL = 11, 12, 13, 20, 28  # kWhereBwd*


@pytest.mark.parametrize("load,wheres,issuer", [
    (1, {LOAD_KV, S_FULL, DQ_FULL, LD_FULL}, None),  # V: every role's first wait begins with the item
    (2, {LOAD_Q}, 0),  # Q rows: the issuer of S^T is the first to wait for them, a step ahead
    (3, {LOAD_Q}, 1),  # dO rows
    (4, {LOAD_Q}, 0),  # dO columns
    (5, {LOAD_Q}, 1),  # Q columns
])
def test_both_ctas_unwind(load, wheres, issuer):
    import torch

    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    env = dict(os.environ, NSP_LIBRARY=str(ROOT / "paper_2609_22755_b200" / "libnsp_checked.so"))
    r = subprocess.run([sys.executable, str(ROOT / "tests" / "withheld_pair_load_case.py"), str(load)], env=env,
                       capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr
    code, item, where, aux = map(int, r.stdout.split("status ")[1].split())
    assert (code, item) == (5, 0) and where in wheres, (code, item, where, aux)  # NSP_ERR_DEVICE_TIMEOUT
    assert issuer is None or aux == issuer
