"""Draws from complex64 states with amplitudes that are not finite, or whose squares
are not: a NaN weighs nothing and leaves the rest as it is, an infinity takes its
group of 2^13 amplitudes' weight with it, squares past FP32's range draw as any
others do."""
import numpy as np
import pytest
import torch

import oracle
from paper_2401_02852_gb300 import api
from paper_2401_02852_gb300 import instances as gen

pytestmark = pytest.mark.gpu

CASES = [(4, [3]), (9, [0, 17, 511]), (13, [0, 5000]), (15, [1, 8191, 20000]), (15, list(range(64, 96)))]


@pytest.mark.parametrize("n,where", CASES)
@pytest.mark.parametrize("value", [complex(np.nan, 0.1), complex(0.1, -np.nan), complex(np.nan, np.nan)])
@pytest.mark.parametrize("aligned", [True, False])
def test_nan_weighs_nothing(n, where, value, aligned):
    psi = gen.random_state("nf", n, 1).astype(np.complex64)
    zero = psi.copy()
    zero[where] = 0
    psi[where] = value
    buf = torch.zeros((1 << n) + 2, dtype=torch.complex64, device="cuda")
    st = buf[2:] if aligned else buf[1:-1]
    st.copy_(torch.from_numpy(psi))
    u = gen.uniforms("nf-u", 4000, n)
    got = api.sample(n, st, u).cpu().numpy()
    assert np.array_equal(got, api.sample(n, torch.from_numpy(zero).cuda(), u).cpu().numpy())
    assert not np.isin(got, where).any()


@pytest.mark.parametrize("n,where", [(14, 100), (15, 8192), (16, 65535)])
def test_an_infinity_takes_its_group(n, where):
    psi = gen.random_state("nf", n, 2).astype(np.complex64)
    zero = psi.copy()
    g = where >> 13
    zero[g << 13:(g + 1) << 13] = 0
    psi[where] = complex(0.0, -np.inf)
    u = gen.uniforms("nf-i", 3000, n)
    got = api.sample(n, torch.from_numpy(psi).cuda(), u).cpu().numpy()
    assert np.array_equal(got, api.sample(n, torch.from_numpy(zero).cuda(), u).cpu().numpy())


def test_an_infinity_beside_squares_past_fp32():
    """All groups' squares overflow, one holds an infinity too: it alone weighs nothing."""
    n = 14
    psi = gen.random_state("nf", n, 4).astype(np.complex64) * np.float32(4e21)
    zero = psi.copy()
    psi[77] = complex(np.inf, 1.0)
    zero[77] = 0
    u = gen.uniforms("nf-b", 3000, n)
    got = api.sample(n, torch.from_numpy(psi).cuda(), u).cpu().numpy()
    assert np.array_equal(got, api.sample(n, torch.from_numpy(zero).cuda(), u).cpu().numpy())


@pytest.mark.parametrize("n", [9, 13, 14])
def test_squares_past_fp32(n):
    psi = gen.random_state("nf", n, 3).astype(np.complex64) * np.float32(4e21 * 2.0 ** ((n - 13) / 2))
    assert np.isfinite(psi).all() and np.abs(psi).max() > 2e19
    p = np.abs(psi.astype(np.complex128)) ** 2
    F = np.cumsum(p.astype(np.longdouble))
    u = gen.uniforms("nf-s", 3000, n)
    got = api.sample(n, torch.from_numpy(psi).cuda(), u).cpu().numpy().astype(np.int64)
    want = oracle.sample(n, psi.astype(np.complex128), u).astype(np.int64)
    for i in np.flatnonzero(got != want):  # equal, but for uniforms within 1e-11 of a step of F
        t = np.longdouble(u[i]) * F[-1]
        for x in (got[i], want[i]):
            assert min(abs(t - (F[x - 1] if x else 0)), abs(t - F[x])) <= 1e-11 * F[-1]
