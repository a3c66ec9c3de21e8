"""A call that the runtime refuses returns its error and leaves nothing behind: the next
call on the same thread is judged by itself."""
import ctypes

import numpy as np
import pytest
import torch


@pytest.mark.gpu
def test_call_after_a_refused_one(lib):
    N = 256
    plan = lib.Plan(N, 25.6, 1, tf32x3=False)
    g = torch.Generator().manual_seed(1)
    x = torch.randn(3, N, generator=g, dtype=torch.float64).cuda()
    want = plan.forward(1, x)
    psi = x.clone()
    U = torch.zeros(N, dtype=torch.float64, device="cuda")
    rt = ctypes.CDLL(f"libcudart.so.{torch.version.cuda.split('.')[0]}")
    st = torch.cuda.Stream()
    ws = torch.empty(plan_states_bytes(lib, plan, 3), dtype=torch.uint8, device="cuda")
    levels = (ctypes.c_double * 3)()
    torch.cuda.synchronize()
    # bound states wait for their result, which a stream that records a graph refuses
    graph = ctypes.c_void_p()
    assert rt.cudaStreamBeginCapture(ctypes.c_void_p(st.cuda_stream), 2) == 0   # relaxed
    rc = lib.load().dsbt_radial_states(plan.handle, 1, U.data_ptr(), 3, 0.05, 1, psi.data_ptr(), levels, None,
                                       ws.data_ptr(), ws.numel(), ctypes.c_void_p(st.cuda_stream))
    left = rt.cudaPeekAtLastError()
    rt.cudaStreamEndCapture(ctypes.c_void_p(st.cuda_stream), ctypes.byref(graph))
    rt.cudaGetLastError()        # of the capture that came to nothing
    assert (rc, left) == (-4, 0)   # DSBT_ERR_CUDA
    assert torch.equal(plan.forward(1, x), want)
    plan.close()


def plan_states_bytes(lib, plan, n):
    return lib.load().dsbt_radial_states_workspace_size(plan.handle, n)
