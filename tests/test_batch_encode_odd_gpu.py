"""Large batches whose variable arrays do not start on a 4-byte boundary."""
import numpy as np
import pytest
import torch

from paper_2401_02852_gb300 import api
from paper_2401_02852_gb300 import instances as gen
from paper_2401_02852_gb300._lib import QaoaError

pytestmark = pytest.mark.gpu


def _insts(odd):
    out = []
    for i, m in enumerate([2000, 2000, 1500, 2100]):
        var, neg = gen.draw_clauses_keys(11, 5, m, gen.rng_for("enc-odd", m, i))
        if i in odd:
            raw = np.zeros(var.nbytes + 4, dtype=np.uint8)
            v = np.ndarray(var.shape, np.int32, buffer=raw, offset=(1 + i - raw.ctypes.data) % 4 or 1)
            v[:] = var
            assert v.flags.c_contiguous and v.ctypes.data % 4
            var = v
        out.append(gen.Instance(n=11, k=5, var=var, neg=neg))
    return out


@pytest.mark.parametrize("odd", [[0], [3], [0, 1, 2]])
def test_tables_of_odd_arrays(odd):
    ref, sols, mx = api.cost_table_batch(_insts([]))
    got, s2, m2 = api.cost_table_batch(_insts(odd))
    assert torch.equal(ref, got) and np.array_equal(sols, s2) and np.array_equal(mx, m2)
    bad = _insts(odd)
    bad[3].var[2000, 4] = 11
    out = torch.full((4, 1 << 11), 77, dtype=torch.uint8, device="cuda")
    with pytest.raises(QaoaError, match="EINVAL: clause 2000"):
        api.cost_table_batch(bad, out=out)
    torch.cuda.synchronize()
    assert bool((out == 77).all())
