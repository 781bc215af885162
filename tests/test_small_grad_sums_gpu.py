"""complex64 gradients of small instances sum p_succ in FP64: with beta = 0 every
solution keeps the amplitude of the initial table, the FP32 number nearest to
2^(-n/2), so p_succ is known up to the rounding of the sum alone (2^n FP64
additions: 1e-12).  FP32 squares or sums are off by about 1e-8 and more."""
import numpy as np
import pytest
import torch

import oracle
from paper_2401_02852_gb300 import api
from paper_2401_02852_gb300 import instances as gen

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [5, 7, 9, 11, 13])
@pytest.mark.parametrize("symmetric", [True, False])
def test_p_succ_of_equal_amplitudes(n, symmetric):
    inst = gen.raw_instance("sums", n, 3, 1.0, 0)
    tab = oracle.cost_table(n, inst.var, inst.neg)[0].astype(np.uint8)
    if not symmetric:
        tab[1] = 1 if tab[1] == 0 else 0
    sols = int(np.sum(tab == 0))
    assert sols > 0
    g, b = np.array([0.3, 0.7, 0.2]), np.zeros(3)
    ps, dg, _ = api.grad(n, torch.from_numpy(tab).cuda(), inst.m, g, b, "c64")
    want = sols * float(np.float32(2.0 ** (-0.5 * n))) ** 2
    assert abs(ps - want) <= 1e-12 * want
    assert np.all(dg == 0.0)
