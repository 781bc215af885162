"""The cooperative evolutions of mid-sized states against the FP64 oracle: every n
of their range (tile sizes 9 to 11, one to three rounds per group), odd and even
depths, full and halved layouts, and the boundary to the HBM passes (batches too
large for the device to hold at once, depth one, n = 21)."""
import numpy as np
import pytest
import torch

import oracle
from paper_2401_02852_gb300 import api
from paper_2401_02852_gb300 import instances as gen
from paper_2401_02852_gb300._lib import DF64, Z2_HALF

pytestmark = pytest.mark.gpu

ARITH = {"c64": ("c64", 0, 1e-6, 1e-4), "c128": ("c128", 0, 2e-15, 1e-10), "df64": ("c128", DF64, 2e-12, 1e-10)}


def _inst(n, m=None):
    inst = gen.raw_instance("mid", n, 5, (m or 4 * n) / n, 0)
    return inst, oracle.cost_table(n, inst.var, inst.neg)[0]


@pytest.mark.parametrize("arith", list(ARITH))
@pytest.mark.parametrize("n,p", [(13, 2), (14, 1), (14, 2), (14, 3), (15, 2), (16, 3), (17, 2), (18, 2), (19, 3), (20, 2),
                                 (21, 2)])
def test_evolution(arith, n, p):
    dtype, flags, tol, ps_tol = ARITH[arith]
    inst, ref = _inst(n)
    g, b = gen.linear_ramp(p)
    b = b * 1.9  # both butterfly forms
    cost, _, _ = api.cost_table(inst)
    psi = oracle.evolve(n, ref, g, b)
    rps, _ = oracle.success_prob(n, ref, psi)
    amp = np.max(np.abs(psi))
    for _ in range(2):  # the barrier words serve launch after launch
        st, ps, nm = api.evolve(n, cost, inst.m, g, b, dtype, flags=flags)
        assert np.max(np.abs(st.cpu().numpy() - psi)) <= tol * (1 + n * p) * amp
        assert abs(ps - rps) <= ps_tol * rps and abs(nm - 1) <= (1e-6 if dtype == "c64" else 1e-10)
    if arith != "df64" and n > (13 if dtype == "c64" else 12):
        half, _, _ = api.cost_table_half(inst)
        sh, ps, nm = api.evolve(n, half, inst.m, g, b, dtype, flags=Z2_HALF)
        assert np.max(np.abs(sh.cpu().numpy() - psi[: 1 << (n - 1)])) <= tol * (1 + n * p) * amp
        assert abs(ps - rps) <= ps_tol * rps and abs(nm - 1) <= (1e-6 if dtype == "c64" else 1e-10)


# the large batches' second group has 1 .. 8 qubits (tiles with rows of 2^12 down to
# 2^5 amplitudes in complex64, 2^11 down to 2^4 in double-float)
@pytest.mark.parametrize("arith,n,small,large", [("c64", 14, 3, 80), ("c64", 15, 1, 40), ("c64", 16, 1, 20),
                                                 ("c64", 17, 1, 12), ("c64", 18, 1, 12), ("c64", 19, 1, 6),
                                                 ("c64", 20, 1, 4), ("c128", 13, 5, 100), ("c128", 17, 1, 12),
                                                 ("df64", 13, 1, 100), ("df64", 14, 1, 60), ("df64", 15, 1, 30),
                                                 ("df64", 16, 2, 12), ("df64", 17, 1, 12), ("df64", 18, 1, 6),
                                                 ("df64", 19, 1, 6), ("df64", 20, 1, 4)])
def test_batch_sizes_on_both_sides(arith, n, small, large):
    """`large` instances do not fit at once and run as HBM passes: the same states
    up to rounding, instance by instance."""
    dtype, flags, tol, ps_tol = ARITH[arith]
    p = 3
    insts = [gen.raw_instance("mid-b", n, 5, 4.0, i) for i in range(small)]
    costs, _, _ = api.cost_table_batch(insts)
    g, b = gen.linear_ramp(p)
    many = costs.repeat((large + small - 1) // small, 1)[:large].contiguous()
    a, pa, _ = api.evolve_batch(n, costs, 4 * n, g, b, dtype, flags=flags)
    c, pc, _ = api.evolve_batch(n, many, 4 * n, g, b, dtype, flags=flags)
    amp = float(a.abs().max())
    for i in range(large):
        assert float((c[i] - a[i % small]).abs().max()) <= 2 * tol * (1 + n * p) * amp
        assert abs(pc[i] - pa[i % small]) <= ps_tol * max(pa[i % small], 1e-30)


def test_long_tables_and_streams():
    """m above 255 (full phase tables), several streams at once, without results."""
    n, p = 15, 4
    inst = gen.raw_instance("mid-l", n, 9, 100.0, 0)
    ref = oracle.cost_table(n, inst.var, inst.neg)[0]
    g, b = gen.linear_ramp(p, scale=0.3)
    cost, _, _ = api.cost_table(inst)
    psi = oracle.evolve(n, ref, g, b)
    streams = [torch.cuda.Stream() for _ in range(4)]
    torch.cuda.synchronize()
    outs = [api.evolve(n, cost, inst.m, g, b, "c64", want=False, stream=s)[0] for s in streams for _ in range(3)]
    torch.cuda.synchronize()
    for o in outs:
        assert np.max(np.abs(o.cpu().numpy() - psi)) <= 1e-6 * (1 + n * p) * np.max(np.abs(psi))
