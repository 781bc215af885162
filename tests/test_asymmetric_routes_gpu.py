"""Tables that are not flip-symmetric on each route of an evolution, the route
itself asserted by the kernels that ran: the cooperative launch at its larger tile
sizes, the HBM passes of one instance (complex64 low passes with three buffers;
initial, phase, fused, plain and reducing passes) and of batches whose last group
has from one qubit to a whole group's.  Against the FP64 oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_2401_02852_gb300 import api
from paper_2401_02852_gb300 import instances as gen
from paper_2401_02852_gb300._lib import DF64

pytestmark = pytest.mark.gpu

ARITH = {"c64": ("c64", 0, 1e-6, 1e-4), "c128": ("c128", 0, 2e-15, 1e-10), "df64": ("c128", DF64, 2e-12, 1e-10)}


def _tables(n, where):
    inst = gen.raw_instance("routes", n, 5, 4.0, 0)
    ref = oracle.cost_table(n, inst.var, inst.neg)[0].astype(np.uint8)
    out = []
    for x in where:
        t = ref.copy()
        if x is not None:
            t[x] = t[x] + 1 if t[x] < inst.m else t[x] - 1
        out.append(t)
    return inst.m, np.stack(out)


def _run(arith, n, p, tabs, m, reps=1):
    dtype, flags, tol, ps_tol = ARITH[arith]
    g, b = gen.linear_ramp(p)
    b = b * 1.5  # both butterfly forms
    costs = torch.from_numpy(tabs).cuda()
    many = costs.repeat(reps, 1).contiguous()
    with api.Profiler() as prof:
        states, ps, nm = api.evolve_batch(n, many, m, g, b, dtype, flags=flags)
    for i, t in enumerate(tabs):
        psi = oracle.evolve(n, t, g, b)
        rps, _ = oracle.success_prob(n, t, psi)
        amp = np.max(np.abs(psi))
        assert np.max(np.abs(states[i].cpu().numpy() - psi)) <= tol * (1 + n * p) * amp
        for j in range(i, many.shape[0], len(tabs)):
            assert torch.equal(states[j], states[i])
            assert abs(ps[j] - rps) <= ps_tol * rps and abs(nm[j] - 1) <= (1e-6 if dtype == "c64" else 1e-10)
    return prof.stats


# tiles of 2^10 and 2^11 amplitudes; the moved entry in the first, a middle and the last tile
@pytest.mark.parametrize("arith", list(ARITH))
@pytest.mark.parametrize("n,p,at", [(17, 2, 0.0), (18, 3, 0.999), (19, 2, 0.3), (19, 3, 0.0), (20, 2, 0.7), (20, 3, 0.999)])
def test_cooperative_launch(arith, n, p, at):
    m, tabs = _tables(n, [int(at * (1 << n))])
    stats = _run(arith, n, p, tabs, m)
    assert "mid" in stats and "pass_low" not in stats


@pytest.mark.parametrize("arith,n,p", [("c64", 21, 1), ("c64", 21, 2), ("c64", 21, 3), ("c64", 22, 2), ("c64", 22, 3),
                                       ("c64", 23, 2), ("c128", 21, 3), ("df64", 21, 3), ("df64", 22, 2)])
def test_passes_of_one_instance(arith, n, p):
    m, tabs = _tables(n, [(1 << n) - 5])
    stats = _run(arith, n, p, tabs, m)
    assert "mid" not in stats and stats["pass_low"][0] >= 1 and stats["flip_check"][0] == 1


# batches that do not fit the device at once: a symmetric and two other tables, repeated
@pytest.mark.parametrize("arith,n,reps", [("c64", 14, 30), ("c64", 15, 16), ("c64", 16, 8), ("c64", 17, 5), ("c64", 18, 5),
                                          ("c64", 19, 3), ("c64", 20, 2), ("df64", 13, 36), ("df64", 14, 22),
                                          ("df64", 15, 11), ("df64", 16, 6), ("df64", 17, 5), ("df64", 18, 3),
                                          ("df64", 19, 3), ("c128", 13, 36), ("c128", 16, 6)])
@pytest.mark.parametrize("p", [2, 3])  # the last pass low and high
def test_passes_of_batches(arith, n, reps, p):
    m, tabs = _tables(n, [None, 3, 3 << (n - 2)])
    stats = _run(arith, n, p, tabs, m, reps)
    assert "mid" not in stats and "pass_high" in stats
