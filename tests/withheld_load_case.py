"""Run by test_gpu_failure_record.py with NSP_LIBRARY pointing at libnsp_checked.so: the record of a wait that runs out names the
wait. One V tile of the first item is never loaded; the MMA issuer reaches that wait first and its limit runs out first."""
import sys
from pathlib import Path

ROOT = Path(__file__).resolve().parent.parent
sys.path.insert(0, str(ROOT))
sys.path.insert(0, str(ROOT / "tests"))

import torch  # noqa: E402

import parity_util as P  # noqa: E402
from paper_2609_22755_b200 import binding as B  # noqa: E402
from paper_2609_22755_b200 import workloads as W  # noqa: E402

FWD_LOAD = 1  # kWhereFwdLoad
for head_dim in (128, 64):
    for _ in range(5):
        run = P.GpuRun(W.custom([500, 300], 4, 2, seed=91, head_dim=head_dim))
        B.nsp_plan_set_wait_limit(run.plan, 2_000_000)
        B.nsp_checked_withhold_load(run.plan, True)
        run.forward()
        torch.cuda.synchronize()  # the launch ends by itself
        code, item, where, aux = B.nsp_device_status(run.plan)
        print("withheld load:", (code, item, where, aux))
        assert code == B.NSP_ERR_DEVICE_TIMEOUT and where == FWD_LOAD, (code, item, where, aux)
