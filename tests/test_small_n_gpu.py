"""The small-n kernels (whole evolutions and gradients in shared memory) against
the FP64 oracle: every n of their range, flip-symmetric and other tables in one
batch, the cluster sizes a batch count selects, tables at odd addresses, tables
and angles too long for kernel parameters."""
import numpy as np
import pytest
import torch

import oracle
from paper_2401_02852_gb300 import api
from paper_2401_02852_gb300 import instances as gen
from paper_2401_02852_gb300._lib import DF64

pytestmark = pytest.mark.gpu

ARITH = {"c64": ("c64", 0, 1e-6, 1e-4), "c128": ("c128", 0, 2e-15, 1e-10), "df64": ("c128", DF64, 2e-12, 1e-10)}


def _tables(n, count):
    """`count` tables of one instance, every second one made asymmetric (one
    entry moved); n < 2 has no clause."""
    k = min(3, n)
    inst = gen.raw_instance("small", n, k, 3.0, 0)
    ref = oracle.cost_table(n, inst.var, inst.neg)[0].astype(np.uint8)
    tabs = np.repeat(ref[None], count, 0)
    rng = np.random.default_rng(n)
    for i in range(1, count, 2):
        x = rng.integers(0, 1 << n)
        tabs[i, x] = tabs[i, x] + 1 if tabs[i, x] < inst.m else tabs[i, x] - 1
    return inst.m, tabs


@pytest.mark.parametrize("arith", list(ARITH))
@pytest.mark.parametrize("n", range(1, 14))
def test_evolutions(arith, n):
    dtype, flags, tol, ps_tol = ARITH[arith]
    if n > (13 if dtype == "c64" else 12):
        pytest.skip("above the one-CTA range of the arithmetic")
    p = 3
    m, tabs = _tables(n, 3)
    g, b = gen.linear_ramp(p)
    b = b * 1.9  # both butterfly forms (beta below and above pi / 4)
    states, ps, nm = api.evolve_batch(n, torch.from_numpy(tabs).cuda(), m, g, b, dtype, flags=flags)
    for i, t in enumerate(tabs):
        psi = oracle.evolve(n, t, g, b)
        rps, _ = oracle.success_prob(n, t, psi)
        assert np.max(np.abs(states[i].cpu().numpy() - psi)) <= tol * (1 + n * p) * np.max(np.abs(psi))
        assert abs(ps[i] - rps) <= ps_tol * rps and abs(nm[i] - 1) <= (1e-6 if dtype == "c64" else 1e-10)


# FP64 batches of these counts take clusters of 8, 4, 2 and 1 CTAs
@pytest.mark.parametrize("n,count", [(12, 1), (12, 100), (11, 40), (12, 60), (12, 160), (10, 20)])
def test_cluster_sizes(n, count):
    p = 2
    m, tabs = _tables(n, count)
    g, b = gen.linear_ramp(p)
    costs = torch.from_numpy(tabs).cuda()
    states, ps, nm = api.evolve_batch(n, costs, m, g, b, "c128")
    gps, dg, db = api.grad_batch(n, costs, m, g, b, "c128")
    for i in sorted({0, 1, count // 2, count - 1} & set(range(count))):
        psi = oracle.evolve(n, tabs[i], g, b)
        rps, rdg, rdb = oracle.grad(n, tabs[i], g, b)
        assert np.max(np.abs(states[i].cpu().numpy() - psi)) <= 2e-15 * (1 + n * p) * np.max(np.abs(psi))
        assert abs(ps[i] - rps) <= 1e-10 * rps and abs(gps[i] - rps) <= 1e-10 * rps and abs(nm[i] - 1) < 1e-12
        scale = max(np.max(np.abs(rdg)), np.max(np.abs(rdb)))
        assert max(np.max(np.abs(dg[i] - rdg)), np.max(np.abs(db[i] - rdb))) <= 1e-8 * scale


@pytest.mark.parametrize("dtype", ["c64", "c128"])
@pytest.mark.parametrize("n", range(1, 14))
def test_gradients(dtype, n):
    if n > (13 if dtype == "c64" else 12):
        pytest.skip("above the one-CTA range of the arithmetic")
    p = 4
    m, tabs = _tables(n, 3)
    g, b = gen.linear_ramp(p)
    b = b * 1.9
    ps, dg, db = api.grad_batch(n, torch.from_numpy(tabs).cuda(), m, g, b, dtype)
    for i, t in enumerate(tabs):
        rps, rdg, rdb = oracle.grad(n, t, g, b)
        scale = max(np.max(np.abs(rdg)), np.max(np.abs(rdb)))
        tol = 1e-6 * (1 + n * p) if dtype == "c64" else 1e-8
        assert abs(ps[i] - rps) <= (1e-4 if dtype == "c64" else 1e-10) * rps
        # at n = 1 the derivatives may all be zero up to rounding
        assert max(np.max(np.abs(dg[i] - rdg)), np.max(np.abs(db[i] - rdb))) <= tol * max(scale, 1.0 if n < 3 else 0.0)


@pytest.mark.parametrize("dtype,n", [("c64", 9), ("c128", 12), ("c64", 13)])
def test_odd_table_address_and_staged_tables(dtype, n):
    """A table that starts at an odd address, m above 255 (full phase tables) and
    p = 20: the tables are staged instead of passed as kernel parameters."""
    p = 20
    m, tabs = _tables(n, 2)
    buf = torch.zeros((2 << n) + 16, dtype=torch.uint8, device="cuda")
    costs = buf[3:3 + (2 << n)].view(2, 1 << n)
    costs.copy_(torch.from_numpy(tabs))
    g, b = gen.linear_ramp(p)
    states, ps, _ = api.evolve_batch(n, costs, 300, g, b, dtype)
    gps, dg, db = api.grad_batch(n, costs, 300, g, b, dtype)
    tol = 1e-6 if dtype == "c64" else 2e-15
    for i, t in enumerate(tabs):
        psi = oracle.evolve(n, t, g, b)
        rps, rdg, rdb = oracle.grad(n, t, g, b)
        assert np.max(np.abs(states[i].cpu().numpy() - psi)) <= tol * (1 + n * p) * np.max(np.abs(psi))
        rel = 1e-4 if dtype == "c64" else 1e-10
        assert abs(ps[i] - rps) <= rel * rps and abs(gps[i] - rps) <= rel * rps
        scale = max(np.max(np.abs(rdg)), np.max(np.abs(rdb)))
        gtol = 1e-6 * (1 + n * p) if dtype == "c64" else 1e-8
        assert max(np.max(np.abs(dg[i] - rdg)), np.max(np.abs(db[i] - rdb))) <= gtol * scale
