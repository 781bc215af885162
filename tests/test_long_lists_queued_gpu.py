"""Clause lists too long for kernel parameters, several in flight: each table is
made from its own list."""
import numpy as np
import pytest

import oracle
from paper_2401_02852_gb300 import instances as gen
from paper_2401_02852_gb300.serve import Server

pytestmark = pytest.mark.gpu


def test_queued_long_lists():
    n, p = 14, 2
    g, b = gen.linear_ramp(p, scale=0.3)
    # one size, different clauses; different angles keep the requests from grouping
    insts = [gen.raw_instance("long-q", n, 9, 1100 / n, i) for i in range(12)]
    assert all(i.m > 1023 for i in insts)
    with Server("c64", small_n_max=13, n_streams=6) as s:
        tickets = [s.submit(inst, g * (1 + 0.01 * i), b) for i, inst in enumerate(insts)]
        res = [s.wait(t) for t in tickets]
        assert s.stats()["single_launches"] == len(insts)
    for i, (inst, r) in enumerate(zip(insts, res)):
        ref, sols, mx = oracle.cost_table(n, inst.var, inst.neg)
        ref_ps, _ = oracle.success_prob(n, ref, oracle.evolve(n, ref, g * (1 + 0.01 * i), b))
        assert r.status == 0 and r.n_sol == sols and r.max_cost == mx
        assert abs(r.p_succ - ref_ps) <= 1e-4 * ref_ps
