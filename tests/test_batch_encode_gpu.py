"""Batched cost tables whose clauses are checked and encoded on the device (2^15
literals and more) against the oracle, around that size and for clause lengths
up to n, and their rejection of invalid literals before anything is written."""
import numpy as np
import pytest
import torch

import oracle
from paper_2401_02852_gb300 import api
from paper_2401_02852_gb300 import instances as gen
from paper_2401_02852_gb300._lib import QaoaError

pytestmark = pytest.mark.gpu


def _insts(n, k, ms):
    out = []
    for i, m in enumerate(ms):
        var, neg = gen.draw_clauses_keys(n, k, m, gen.rng_for("enc", n, k, m, i))
        out.append(gen.Instance(n=n, k=k, var=var, neg=neg))
    return out


# 2^15 literals are 6554 clauses of 5: just below, just above; ragged lists with
# empty ones; single-literal clauses; clauses over all variables; 9-literal lists
# past 1023 clauses
@pytest.mark.parametrize("n,k,ms", [(10, 5, [3276, 3277]), (10, 5, [3277, 3277]), (9, 3, [0, 5000, 257, 0, 6000]),
                                    (7, 1, [8000, 8000, 8000, 8000, 800]), (9, 9, [1000, 2000, 900]),
                                    (13, 9, [3000, 1023, 1024, 1])])
def test_tables_match_oracle(n, k, ms):
    insts = _insts(n, k, ms)
    out = torch.zeros((len(ms), 1 << n), dtype=torch.uint8, device="cuda")
    refs = [oracle.cost_table(n, i.var, i.neg) if i.m else (np.zeros(1 << n, np.uint16), 1 << n, 0) for i in insts]
    if max(r[2] for r in refs) > 255:  # the call reports it, the tables hold the counts mod 256
        with pytest.raises(QaoaError):
            api.cost_table_batch(insts, out=out)
    else:
        _, sols, mxs = api.cost_table_batch(insts, out=out)
        assert [int(s) for s in sols] == [r[1] for r in refs] and [int(m) for m in mxs] == [r[2] for r in refs]
    for t, r in zip(out.cpu().numpy(), refs):
        assert np.array_equal(t, (r[0] % 256).astype(np.uint8))


def test_read_only_and_foreign_arrays():
    insts = _insts(11, 5, [2000] * 4)
    ref, _, _ = api.cost_table_batch(insts)
    ro = [gen.Instance(n=i.n, k=i.k, var=np.asfortranarray(i.var).astype(np.int64), neg=i.neg.copy()) for i in insts]
    for i in ro:
        i.var.flags.writeable = False
        i.neg.flags.writeable = False
    got, _, _ = api.cost_table_batch(ro)
    assert torch.equal(ref, got)


@pytest.mark.parametrize("bad", ["high", "negative", "flag", "repeated"])
def test_invalid_literals_are_refused(bad):
    insts = _insts(10, 5, [4000, 4000])
    v, g = insts[1].var, insts[1].neg
    if bad == "high":
        v[3999, 4] = 10
    elif bad == "negative":
        v[17, 0] = -3
    elif bad == "flag":
        g[255, 2] = 2
    else:
        v[256, 1] = v[256, 3]
    out = torch.full((2, 1 << 10), 77, dtype=torch.uint8, device="cuda")
    with pytest.raises(QaoaError, match="EINVAL: clause"):
        api.cost_table_batch(insts, out=out)
    torch.cuda.synchronize()
    assert bool((out == 77).all())
