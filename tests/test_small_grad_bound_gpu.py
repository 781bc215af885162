"""Gradients of small instances whose table exceeds the given clause count: costs
above m count as m, in the phases and in the derivatives."""
import numpy as np
import pytest
import torch

import oracle
from paper_2401_02852_gb300 import api
from paper_2401_02852_gb300 import instances as gen

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,n,count", [("c64", 4, 1), ("c64", 13, 2), ("c128", 12, 1), ("c128", 11, 40), ("c128", 9, 2)])
def test_costs_above_m(dtype, n, count):
    p, m = 3, 2
    inst = gen.raw_instance("bound", n, 3, 1.5, 0)
    tab = oracle.cost_table(n, inst.var, inst.neg)[0].astype(np.uint8)
    assert tab.max() > m and (tab == 0).any()
    g, b = gen.linear_ramp(p)
    ps, dg, db = api.grad_batch(n, torch.from_numpy(np.repeat(tab[None], count, 0)).cuda(), m, g, b, dtype)
    rps, rdg, rdb = oracle.grad(n, np.minimum(tab, m), g, b)
    scale = max(np.max(np.abs(rdg)), np.max(np.abs(rdb)))
    tol = 1e-6 * (1 + n * p) if dtype == "c64" else 1e-8
    for i in range(count):
        assert abs(ps[i] - rps) <= (1e-4 if dtype == "c64" else 1e-10) * rps
        assert max(np.max(np.abs(dg[i] - rdg)), np.max(np.abs(db[i] - rdb))) <= tol * scale
