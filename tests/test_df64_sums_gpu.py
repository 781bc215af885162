"""p_succ of double-float evolutions when many amplitudes of a thread are solutions:
with p = 0 all amplitudes are equal, and 16 equal terms sum exactly (pairwise, or
compensated), so with every x a solution p_succ is the norm to the last bit."""
import numpy as np
import pytest
import torch

import oracle
from paper_2401_02852_gb300 import api
from paper_2401_02852_gb300 import instances as gen
from paper_2401_02852_gb300._lib import DF64

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [13, 15, 21, 23])
def test_equal_amplitudes(n):
    cost = torch.zeros(1 << n, dtype=torch.uint8, device="cuda")
    _, ps, nm = api.evolve(n, cost, 0, [], [], "c128", flags=DF64)
    assert ps == nm and abs(nm - 1) <= 1e-12


@pytest.mark.parametrize("n,p", [(21, 1), (21, 2), (22, 3)])
def test_dense_solutions(n, p):
    """One x in two is a solution, in the passes' last low and last high pass."""
    rng = np.random.default_rng(n)
    half = (rng.random(1 << (n - 1)) < 0.5).astype(np.uint8)
    tab = np.concatenate([half, half[::-1]])
    g, b = gen.linear_ramp(p)
    psi = oracle.evolve(n, tab, g, b)
    rps, _ = oracle.success_prob(n, tab, psi)
    st, ps, nm = api.evolve(n, torch.from_numpy(tab).cuda(), 1, g, b, "c128", flags=DF64)
    assert abs(ps - rps) <= 1e-10 * rps and abs(nm - 1) <= 1e-10
    # against the stored state's own sum, 2^21 FP64 terms pairwise on both sides
    w = st.real.square() + st.imag.square()
    mine = float((w * torch.from_numpy(tab == 0).cuda()).sum())
    assert abs(ps - mine) <= 1e-14 * mine
