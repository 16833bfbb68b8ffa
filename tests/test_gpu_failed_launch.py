"""A launch that fails is reported by its own call and by no later one."""
import ctypes

import pytest

pytestmark = pytest.mark.gpu


def test_error_of_a_failed_launch_does_not_stay_behind():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2609_22755_b200 import binding as B

    x = torch.zeros(4 * 8 * 64, dtype=torch.bfloat16, device="cuda")
    y = torch.empty_like(x)
    B.nsp_plan_tiles([0, 200], [4], [2]).destroy()
    torch.cuda.synchronize()
    with open("/proc/self/maps") as f:
        path = next(line.split()[-1] for line in f if "libcudart" in line)
    rt = ctypes.CDLL(path)
    s = torch.cuda.Stream()
    handle = ctypes.c_void_p(s.cuda_stream)
    assert rt.cudaStreamBeginCapture(handle, 1) == 0  # thread-local mode
    assert rt.cudaStreamSynchronize(handle) != 0  # not allowed under capture: the capture is no longer valid
    with pytest.raises(B.NspError):  # and a launch into it fails on the host
        B.nsp_a2a_gather_heads(x, y, 4, 8, 4, 64, [0, 4], stream=s)
    graph = ctypes.c_void_p()
    assert rt.cudaStreamEndCapture(handle, ctypes.byref(graph)) != 0
    rt.cudaGetLastError()
    B.nsp_plan_tiles([0, 200], [4], [2])
    B.nsp_a2a_gather_heads(x, y, 4, 8, 4, 64, [0, 4], stream=s)
    s.synchronize()
    assert torch.equal(x, y)
