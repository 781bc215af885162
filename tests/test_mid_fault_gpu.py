"""A grid barrier that ran out of time after its call returned: the kernel's word is
set here from the host, as the kernel sets it (no launch is made to fail).  The
next call on that stream reports it, once, and the stream works again."""
import ctypes

import numpy as np
import pytest
import torch

import oracle
from paper_2401_02852_gb300 import _lib, api
from paper_2401_02852_gb300 import instances as gen
from paper_2401_02852_gb300._lib import QaoaError

pytestmark = pytest.mark.gpu


def _word(stream):
    """The stream's fault word (qaoa::fault_word)."""
    f = _lib.load()["_ZN4qaoa10fault_wordEP11CUstream_stPPi"]
    out = ctypes.POINTER(ctypes.c_int)()
    assert f(ctypes.c_void_p(stream.cuda_stream), ctypes.byref(out)) == 0
    return out


def _calls(n, cost, inst, state, g, b, s):
    u = torch.rand(16, dtype=torch.float64, device="cuda")
    return {
        "evolve": lambda: api.evolve(n, cost, inst.m, g, b, "c64", out=state, stream=s),
        "queued evolve": lambda: api.evolve(n, cost, inst.m, g, b, "c64", out=state, want=False, stream=s),
        "table": lambda: api.cost_table(inst, stream=s),
        "gradient": lambda: api.grad(n, cost, inst.m, g, b, "c64", stream=s),
        "success": lambda: api.success_prob(n, cost, state, stream=s),
        "sample": lambda: api.sample(n, state, u, stream=s),
        "running time": lambda: api.running_time(n, cost, state, u, stream=s),
    }


CALLS = ["evolve", "queued evolve", "table", "gradient", "success", "sample", "running time"]


@pytest.mark.parametrize("call", CALLS)
def test_next_call_reports_a_queued_failure_once(call):
    n = 15
    inst = gen.raw_instance("mid-f", n, 5, 4.0, 0)
    ref = oracle.cost_table(n, inst.var, inst.neg)[0]
    g, b = gen.linear_ramp(3)
    cost, _, _ = api.cost_table(inst)
    s, other = torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()
    state, ps, _ = api.evolve(n, cost, inst.m, g, b, "c64", stream=s)
    assert abs(ps - oracle.success_prob(n, ref, oracle.evolve(n, ref, g, b))[0]) <= 1e-4 * ps
    run = _calls(n, cost, inst, state, g, b, s)[call]
    run()
    s.synchronize()
    word = _word(s)
    assert word[0] == 0
    word[0] = 1
    assert api.evolve(n, cost, inst.m, g, b, "c64", stream=other)[1] == ps  # other streams go on
    with pytest.raises(QaoaError, match="grid barrier"):
        run()
    assert word[0] == 0
    run()
    assert api.evolve(n, cost, inst.m, g, b, "c64", stream=s)[1] == ps


def test_failure_while_the_success_probability_waits():
    """The word is set while the reduction is queued behind other work."""
    n = 15
    inst = gen.raw_instance("mid-f", n, 5, 4.0, 0)
    g, b = gen.linear_ramp(3)
    cost, _, _ = api.cost_table(inst)
    s = torch.cuda.Stream()
    torch.cuda.synchronize()
    state, ps, _ = api.evolve(n, cost, inst.m, g, b, "c64", stream=s)
    word = _word(s)
    one = torch.ones(1, dtype=torch.int32).pin_memory()
    view = torch.from_numpy(np.ctypeslib.as_array(word, shape=(1,)))
    api.success_prob(n, cost, state, stream=s)
    for fn in ("qaoa_success_prob", "qaoa_success_prob_noalloc"):
        with torch.cuda.stream(s):
            torch.cuda._sleep(100_000_000)
            dev = one.to("cuda", non_blocking=True)
            view.copy_(dev, non_blocking=True)  # pinned destination: stream ordered
        out = ctypes.c_double(), ctypes.c_double()
        rc = getattr(_lib.load(), fn)(n, ctypes.c_void_p(cost.data_ptr()), ctypes.c_void_p(state.data_ptr()), _lib.C64,
                                      ctypes.byref(out[0]), ctypes.byref(out[1]), ctypes.c_void_p(s.cuda_stream))
        assert rc == -4 and word[0] == 0
        assert abs(api.success_prob(n, cost, state, stream=s)[0] - ps) <= 1e-6 * ps
