"""Requests of one to four variables packed together with larger ones: tables of
fewer than 16 bytes come before tables written 16 bytes at a time."""
import numpy as np
import pytest

import oracle
from paper_2401_02852_gb300 import instances as gen
from paper_2401_02852_gb300.serve import Server

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["c64", "c128"])
def test_tiny_requests_between_larger_ones(dtype):
    sizes = [3, 12, 1, 5, 2, 6, 1, 1, 9, 4, 3, 8, 2, 10]
    p = 3
    g, b = gen.linear_ramp(p)
    insts = [gen.raw_instance("tiny", n, min(3, n), 2.0, i) for i, n in enumerate(sizes)]
    with Server(dtype, n_streams=1) as s:
        big = gen.raw_instance("tiny", 22, 3, 2.0, 99)  # holds the slot while the others queue
        first = s.submit(big, *gen.linear_ramp(20))
        tickets = [s.submit(i, g, b) for i in insts]
        assert s.wait(first).status == 0
        res = [s.wait(t) for t in tickets]
    for inst, r in zip(insts, res):
        ref, sols, mx = oracle.cost_table(inst.n, inst.var, inst.neg)
        rps, _ = oracle.success_prob(inst.n, ref, oracle.evolve(inst.n, ref, g, b))
        assert r.status == 0 and r.n_sol == sols and r.max_cost == mx
        assert abs(r.p_succ - rps) <= (1e-4 if dtype == "c64" else 1e-10) * max(rps, 1e-12)
        assert abs(r.norm - 1) <= (1e-6 if dtype == "c64" else 1e-10)
