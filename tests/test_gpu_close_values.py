"""FP64 calls whose wanted singular values lie close together: the refinement of
the l x l core leaves such pairs to Jacobi sweeps, which keep the basis they
are given as orthonormal as it was.

Tolerances: orthonormality and parity with the exact rank-k part 1e-12, as for
every FP64 call (some ten sweeps of 255 rotations of a column: 1e-13 at l =
256); the Nystrom eigenvalues 1e-10 and product 1e-9, as in its other tests.
"""

import numpy as np
import pytest
import torch

import synth
from oracle import lowrank as orc

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib():
    import paper_2210_11295_gb300 as m

    return m


def _spectrum(l, spread, rng):
    """l values: half of them 1 to 1 + spread, the rest decaying from 0.5."""
    h = l // 2
    return np.sort(np.concatenate([1.0 + spread * rng.random(h), 0.5 * np.exp(-6.0 * np.arange(l - h) / l)]))[::-1]


def _pairs(l, rng):
    """l values in pairs 1e-4 to 1e-15 apart."""
    base = np.exp(-4.0 * np.arange(l // 2) / (l // 2))
    return np.sort(np.concatenate([base, base * (1.0 + 10.0 ** -rng.uniform(4, 15, l // 2))]))[::-1]


def _orth_error(x):
    return np.linalg.norm(x.T @ x - np.eye(x.shape[1]), 2)


@pytest.mark.parametrize("l", [80, 160, 256])
@pytest.mark.parametrize("spread", [1e-3, 1e-4, 1e-5, 1e-6, 0.0, "pairs"])
def test_rsvd_close_values(lib, l, spread):
    rng = np.random.default_rng(l)
    sigma = _pairs(l, rng) if spread == "pairs" else _spectrum(l, spread, rng)
    n, m, k = 8192, l + 13, l // 2
    uu, vv = synth.haar(n, l, rng), synth.haar(m, l, rng)
    a = np.ascontiguousarray((uu * sigma) @ vv.T)
    u, s, v = (x.cpu().numpy() for x in lib.bsrht_rsvd(torch.from_numpy(a).cuda(), k, l, 16, 3))
    assert _orth_error(v) <= 1e-12
    assert _orth_error(u) <= 1e-12
    assert np.max(np.abs(s - sigma[:k])) <= 1e-12 * sigma[0]
    assert np.linalg.norm(a @ v - u * s) <= 1e-12 * np.linalg.norm(a)
    assert np.linalg.norm(a.T @ u - v * s) <= 1e-12 * np.linalg.norm(a)


@pytest.mark.parametrize("l,spread", [(80, 1e-4), (160, 1e-5), (256, 1e-6), (160, "pairs")])
def test_nystrom_close_values(lib, l, spread):
    rng = np.random.default_rng(l)
    lam = _pairs(l, rng) if spread == "pairs" else _spectrum(l, spread, rng)
    n, k = 1536, l // 2
    q = synth.haar(n, l, rng)
    a = (q * lam) @ q.T
    a = np.ascontiguousarray(0.5 * (a + a.T))
    u, got = (x.cpu().numpy() for x in lib.bsrht_nystrom(torch.from_numpy(a).cuda(), k, l, 16, 3))
    assert _orth_error(u) <= 1e-12
    assert np.max(np.abs(got - lam[:k])) <= 1e-7 * lam[0]
    assert np.linalg.norm(a @ u - u * got) <= 1e-7 * np.linalg.norm(a)


@pytest.mark.parametrize("l,decay", [(80, 4.0), (128, 8.0), (300, 15.0), (700, 40.0)])
def test_rsvd_core_singular_in_fp32(lib, l, decay):
    """exp(-i / decay): the l x l core reaches below FP32's rounding of its
    largest value (2e-9 to 2.5e-8), so its FP32 phase gives no basis.  (Omega has
    a repeated row at l = 300 and 700: the rank-k part is the oracle's, off A's
    by 3e-9 and 3e-8.)"""
    rng = np.random.default_rng(l)
    sigma = np.exp(-np.arange(l) / decay)
    n, m, k = 8192, l + 13, 20
    uu, vv = synth.haar(n, l, rng), synth.haar(m, l, rng)
    a = np.ascontiguousarray((uu * sigma) @ vv.T)
    u, s, v = (x.cpu().numpy() for x in lib.bsrht_rsvd(torch.from_numpy(a).cuda(), k, l, 16, 3))
    assert _orth_error(v) <= 1e-12
    assert _orth_error(u) <= 1e-12
    assert np.max(np.abs(s - sigma[:k])) <= 1e-12
    ur, sr, vr = orc.rsvd(a, k, l, 16, 3)
    ref = (ur * sr) @ vr.T
    assert np.linalg.norm((u * s) @ v.T - ref) <= 1e-12 * np.linalg.norm(ref)


@pytest.mark.parametrize("l,spread", [(80, 1e-4), (160, 1e-6), (256, 0.0), (300, "steep")])
def test_rsvd_fp32_data(lib, l, spread):
    """The same cores from FP32 data, whose FP64 polish stops at 16 sqrt(l) 2^-40
    and whose tall factors are accurate to FP32: 1e-5, V orthonormal to 1e-12, U to
    1e-4 as for FP32 data elsewhere."""
    rng = np.random.default_rng(l)
    sigma = np.exp(-np.arange(l) / 15.0) if spread == "steep" else _spectrum(l, spread, rng)
    n, m, k = 8192, l + 13, 20 if spread == "steep" else l // 2
    uu, vv = synth.haar(n, l, rng), synth.haar(m, l, rng)
    x = torch.from_numpy((uu * sigma) @ vv.T).float()
    a = x.double().numpy()
    u, s, v = (t.cpu().numpy() for t in lib.bsrht_rsvd(x.cuda(), k, l, 16, 3))
    assert _orth_error(v) <= 1e-12
    assert _orth_error(u) <= 1e-4
    assert np.max(np.abs(s - sigma[:k])) <= 1e-5 * sigma[0]
    assert np.linalg.norm(a @ v - u * s) <= 1e-5 * np.linalg.norm(a)
    assert np.linalg.norm(a.T @ u - v * s) <= 1e-5 * np.linalg.norm(a)
