"""Full-state evolutions take the half of a flip-symmetric table, decided on the
device per instance: against the FP64 oracle for symmetric tables and for tables
with one entry changed anywhere (which must take every amplitude)."""
import numpy as np
import pytest
import torch

import oracle
from paper_2401_02852_gb300 import api
from paper_2401_02852_gb300 import instances as gen
from paper_2401_02852_gb300._lib import DF64

pytestmark = pytest.mark.gpu

ARITH = {"c64": ("c64", 0, 1e-6), "c128": ("c128", 0, 2e-15), "df64": ("c128", DF64, 2e-12)}


def _tables(n, m, where):
    """One instance's table per entry of `where`: unchanged (None), or with the
    entry at that index moved by one."""
    inst = gen.raw_instance("flip", n, 5, m / n, 0)
    ref, _, _ = oracle.cost_table(n, inst.var, inst.neg)
    out = []
    for x in where:
        t = ref.astype(np.uint8).copy()
        if x is not None:
            t[x] = t[x] + 1 if t[x] < inst.m else t[x] - 1
        out.append(t)
    return inst, np.stack(out)


def _check(n, tab, st, ps, nm, g, b, tol):
    psi = oracle.evolve(n, tab, g, b)
    rps, _ = oracle.success_prob(n, tab, psi)
    p = len(g)
    assert np.max(np.abs(st - psi)) <= tol * (1 + n * p) * np.max(np.abs(psi))
    assert abs(ps - rps) <= (1e-4 if tol == 1e-6 else 1e-10) * rps
    assert abs(nm - 1.0) <= (1e-6 if tol == 1e-6 else 1e-10)


# smallest pass sizes (one or two tiles per half), one and two high groups, the
# last pass low (even p, one group) and high
@pytest.mark.parametrize("arith,n,p", [("c64", 14, 2), ("c64", 14, 1), ("c64", 15, 3), ("c64", 18, 2), ("c64", 23, 1),
                                       ("c128", 13, 1), ("c128", 13, 2), ("c128", 16, 3), ("c128", 21, 2),
                                       ("df64", 13, 2), ("df64", 14, 1), ("df64", 17, 2), ("df64", 21, 2)])
def test_mixed_batch_of_symmetric_and_other_tables(arith, n, p):
    dtype, flags, tol = ARITH[arith]
    N = 1 << n
    where = [None, 0, None, N - 1, N // 2 - 1, N // 2, 5 * N // 8 + 3]
    inst, tabs = _tables(n, 4 * n, where)
    g, b = gen.linear_ramp(p)
    g = g + 0.1
    costs = torch.from_numpy(tabs).cuda()
    states, ps, nm = api.evolve_batch(n, costs, inst.m, g, b, dtype, flags=flags)
    got = states.cpu().numpy()
    for i, x in enumerate(where):
        if i != 2:
            _check(n, tabs[i], got[i].astype(np.complex128), ps[i], nm[i], g, b, tol)
    assert np.array_equal(got[0], got[2])
    # a symmetric table's two halves are each other's mirror to the last bit
    assert np.array_equal(got[0], got[0][::-1])


@pytest.mark.parametrize("arith,n", [("c64", 16), ("c128", 14), ("df64", 14)])
def test_single_and_without_results(arith, n):
    """One instance, alone: with and without the host results, on a side stream."""
    dtype, flags, tol = ARITH[arith]
    inst, tabs = _tables(n, 3 * n, [None, 77])
    g, b = gen.linear_ramp(3)
    for t in tabs:
        cost = torch.from_numpy(t).cuda()
        st, ps, nm = api.evolve(n, cost, inst.m, g, b, dtype, flags=flags)
        _check(n, t, st.cpu().numpy().astype(np.complex128), ps, nm, g, b, tol)
        s = torch.cuda.Stream()
        s.wait_stream(torch.cuda.current_stream())
        st2, _, _ = api.evolve(n, cost, inst.m, g, b, dtype, flags=flags, want=False, stream=s)
        s.synchronize()
        assert torch.equal(st, st2)


# one and two high groups, full, partial and top-only masks of the backward plan
@pytest.mark.parametrize("dtype,n,p", [("c64", 14, 2), ("c64", 15, 1), ("c64", 18, 2), ("c64", 20, 3), ("c64", 21, 2),
                                       ("c128", 13, 2), ("c128", 14, 1), ("c128", 19, 2)])
def test_gradients_of_symmetric_and_other_tables(dtype, n, p):
    N = 1 << n
    where = [None, 1, N - 2]
    inst, tabs = _tables(n, 4 * n, where)
    g, b = gen.linear_ramp(p)
    g = g + 0.1
    tdt = torch.complex64 if dtype == "c64" else torch.complex128
    work = tuple(torch.full((len(where), N), 7.0, dtype=tdt, device="cuda") for _ in range(2))
    ps, dg, db = api.grad_batch(n, torch.from_numpy(tabs).cuda(), inst.m, g, b, dtype, work=work)
    tol = 1e-6 * (1 + n * p) if dtype == "c64" else 1e-8
    for i, t in enumerate(tabs):
        rps, rdg, rdb = oracle.grad(n, t, g, b)
        scale = max(np.max(np.abs(rdg)), np.max(np.abs(rdb)))
        assert abs(ps[i] - rps) <= (1e-4 if dtype == "c64" else 1e-10) * rps
        assert np.max(np.abs(dg[i] - rdg)) <= tol * scale and np.max(np.abs(db[i] - rdb)) <= tol * scale
        # the sweep ends on |+>^n, in both halves
        psi = work[0][i].cpu().numpy()
        amp = 2.0 ** (-n / 2)
        assert np.max(np.abs(psi - amp)) <= (2e-6 if dtype == "c64" else 4e-15) * (1 + n * p) * amp
    if dtype == "c64" or n < 19:
        lam = work[1][0]
        assert torch.equal(lam, lam.flip(0))
