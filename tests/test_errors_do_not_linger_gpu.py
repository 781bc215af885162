"""A CUDA call that fails (here: in a stream capture that a synchronising call has
invalidated) is reported by the call it failed in, not by the next valid one."""
import ctypes

import pytest
import torch

from paper_2401_02852_gb300 import api
from paper_2401_02852_gb300 import instances as gen
from paper_2401_02852_gb300._lib import QaoaError

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,dtype", [(12, "c128"), (12, "c64"), (16, "c64"), (21, "c64")])
def test_valid_call_after_a_failed_one(n, dtype):
    rt = ctypes.CDLL("libcudart.so.13")
    inst = gen.raw_instance("linger", n, 3, 2.0, 0)
    g, b = gen.linear_ramp(2)
    cost, _, _ = api.cost_table(inst)
    s = torch.cuda.Stream()
    torch.cuda.synchronize()
    out, ps, _ = api.evolve(n, cost, inst.m, g, b, dtype, stream=s)  # scratch and kernels loaded
    s.synchronize()
    handle = ctypes.c_void_p(s.cuda_stream)
    assert rt.cudaStreamBeginCapture(handle, 2) == 0  # relaxed
    with pytest.raises(QaoaError, match="ECUDA"):
        api.evolve(n, cost, inst.m, g, b, dtype, out=out, stream=s)  # waits for its results
    with pytest.raises(QaoaError, match="ECUDA"):
        api.evolve(n, cost, inst.m, g, b, dtype, out=out, want=False, stream=s)
    assert rt.cudaPeekAtLastError() == 0
    graph = ctypes.c_void_p()
    assert rt.cudaStreamEndCapture(handle, ctypes.byref(graph)) != 0
    rt.cudaGetLastError()  # this test's own call failed
    api.evolve(n, cost, inst.m, g, b, dtype, out=out, want=False, stream=s)  # checks its launches
    assert api.evolve(n, cost, inst.m, g, b, dtype, out=out, stream=s)[1] == ps
