"""Run by test_gpu_pair_failure.py with NSP_LIBRARY pointing at libnsp_checked.so: a wait of the CTA-pair kernel runs out. One
tile of the second CTA never arrives; all roles of both CTAs unwind, the launch ends, the plan refuses further work, and a fresh
plan on the same context gives what a healthy one gave before. argv[1]: the load that is left out."""
import sys
from pathlib import Path

ROOT = Path(__file__).resolve().parent.parent
sys.path.insert(0, str(ROOT))
sys.path.insert(0, str(ROOT / "tests"))

import numpy as np  # noqa: E402
import torch  # noqa: E402

import parity_util as P  # noqa: E402
from paper_2609_22755_b200 import binding as B  # noqa: E402
from paper_2609_22755_b200 import workloads as W  # noqa: E402

w = W.custom([2049] * 20, 16, 4, seed=47)
host = W.make_tensors(w)


def healthy():
    run = P.GpuRun(w, tensors=host, dq_dtype="f32")
    assert B.nsp_plan_pair_items(run.plan)[0] > 0
    run.forward()
    run.backward()
    assert run.status() == (0, 0, 0, 0), run.status()
    return run.results()


want = healthy()
run = P.GpuRun(w, tensors=host, dq_dtype="f32")
run.forward()
B.nsp_plan_set_wait_limit(run.plan, 2_000_000)
B.nsp_checked_withhold_pair_load(run.plan, int(sys.argv[1]))
run.backward()
torch.cuda.synchronize()  # the launch ends by itself
try:
    run.backward()
    raise SystemExit("the plan accepted work after a device-side timeout")
except B.NspError as e:
    assert e.code == B.NSP_ERR_DEVICE_TIMEOUT, e
run.check_guards()
print("status", *B.nsp_device_status(run.plan))
del run
got = healthy()
for n in ("dk", "dv"):
    assert np.array_equal(got[n], want[n]), n
assert np.max(np.abs(got["dq"] - want["dq"])) <= 2e-5 * np.max(np.abs(want["dq"]))  # arrival order, as in the pair tests
