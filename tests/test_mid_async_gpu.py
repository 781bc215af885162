"""Mid-sized evolutions without results return before the stream's earlier work is
done, and each works on its own angles however many are queued."""
import numpy as np
import pytest
import torch

import oracle
from paper_2401_02852_gb300 import api
from paper_2401_02852_gb300 import instances as gen

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("p,m", [(2, 20), (12, 400)])  # tables of a kilobyte, and of 24 KiB
def test_queued_calls_keep_their_tables(p, m):
    """Six calls of one size, each with its own angles, queued behind half a second
    of other work: none waits for it, none reads another call's tables."""
    n, calls = 14, 6
    inst = gen.raw_instance("mid-a", n, 5, m / n, 0)
    ref = oracle.cost_table(n, inst.var, inst.neg)[0]
    cost, _, _ = api.cost_table(inst)
    angles = [gen.linear_ramp(p, scale=0.2 + 0.1 * i) for i in range(calls)]
    s = torch.cuda.Stream()
    api.evolve(n, cost, inst.m, *angles[0], "c64", stream=s)  # scratch and kernels loaded
    outs = [torch.empty(1 << n, dtype=torch.complex64, device="cuda") for _ in range(calls)]
    torch.cuda.synchronize()
    with torch.cuda.stream(s):
        torch.cuda._sleep(1_000_000_000)
    for o, (g, b) in zip(outs, angles):
        api.evolve(n, cost, inst.m, g, b, "c64", want=False, out=o, stream=s)
    assert not s.query()
    s.synchronize()
    for o, (g, b) in zip(outs, angles):
        psi = oracle.evolve(n, ref, g, b)
        assert np.max(np.abs(o.cpu().numpy() - psi)) <= 1e-6 * (1 + n * p) * np.max(np.abs(psi))


def test_more_calls_than_upload_buffers():
    n, p, calls = 14, 3, 40
    inst = gen.raw_instance("mid-a", n, 5, 4.0, 1)
    ref = oracle.cost_table(n, inst.var, inst.neg)[0]
    cost, _, _ = api.cost_table(inst)
    angles = [gen.linear_ramp(1 + i % p, scale=0.2 + 0.02 * i) for i in range(calls)]
    s = torch.cuda.Stream()
    torch.cuda.synchronize()
    outs = [api.evolve(n, cost, inst.m, g, b, "c128", want=False, stream=s)[0] for g, b in angles]
    s.synchronize()
    for o, (g, b) in zip(outs, angles):
        psi = oracle.evolve(n, ref, g, b)
        assert np.max(np.abs(o.cpu().numpy() - psi)) <= 2e-15 * (1 + n * p) * np.max(np.abs(psi))
