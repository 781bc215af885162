"""Draws at the edges of the draw kernel's shapes: states smaller than one lane's
share, than an entry and than a group, states of one and two groups, draw counts
around a warp's and a block's, states scaled far up and down (the group scales at
and past their limits), an unaligned state."""
import numpy as np
import pytest
import torch

import oracle
from paper_2401_02852_gb300 import api
from paper_2401_02852_gb300 import instances as gen

pytestmark = pytest.mark.gpu


def _same_or_tie(psi, u, got, want):
    """Equal draws, except for uniforms within 1e-11 of a step of the exact
    cumulative distribution next to either draw."""
    F = np.cumsum((np.abs(psi.astype(np.complex128)) ** 2).astype(np.longdouble))
    got, want = got.astype(np.int64), want.astype(np.int64)
    for i in np.flatnonzero(got != want):
        t = np.longdouble(u[i]) * F[-1]
        for x in (got[i], want[i]):
            assert min(abs(t - (F[x - 1] if x else 0)), abs(t - F[x])) <= 1e-11 * F[-1]


@pytest.mark.parametrize("dtype", [np.complex64, np.complex128])
@pytest.mark.parametrize("n", [1, 2, 3, 4, 5, 6, 9, 12, 13, 14])
def test_small_states(n, dtype):
    psi = gen.random_state("edge", n, n, sparsity=0.2 if n > 4 else 0.0).astype(dtype)
    st = torch.from_numpy(psi).cuda()
    for k in (1, 7, 8, 63, 64, 65, 1000):
        u = gen.uniforms("edge-u", k, n)
        want = oracle.sample(n, psi.astype(np.complex128), u)
        _same_or_tie(psi, u, api.sample(n, st, u).cpu().numpy(), want)


@pytest.mark.parametrize("scale", [1e-15, 1e-12, 1e12, 1e18])
def test_scaled_states(scale):
    """Draws do not depend on the state's norm, as far as its squares are
    representable: every probability scales alike."""
    n = 13
    psi = gen.random_state("edge", n, 1).astype(np.complex64) * np.float32(scale)
    u = gen.uniforms("edge-s", 500, 2)
    want = oracle.sample(n, psi.astype(np.complex128), u)
    _same_or_tie(psi, u, api.sample(n, torch.from_numpy(psi).cuda(), u).cpu().numpy(), want)


def test_unaligned_state_and_block_edges():
    n = 14
    psi = gen.random_state("edge", n, 3).astype(np.complex64)
    buf = torch.zeros((1 << n) + 1, dtype=torch.complex64, device="cuda")
    buf[1:].copy_(torch.from_numpy(psi))
    u = gen.uniforms("edge-b", 4097, 4)
    a = api.sample(n, buf[1:], u)
    assert torch.equal(a, api.sample(n, torch.from_numpy(psi).cuda(), u))
    _same_or_tie(psi, u, a.cpu().numpy(), oracle.sample(n, psi.astype(np.complex128), u))
