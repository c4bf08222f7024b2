"""Products on 16-bit slices (FP64 in seven digits, 16-bit A against three
slices) through the low-rank calls that use them, at the edges of their tiles
(128 rows, 64 or up to 256 columns, 32 / 64 of K) and of their rules.

Tolerances: FP64 parity 1e-12 (a product is off by at most K 2^-54 times the
largest entries, 3e-13 at the longest K here); FP32 arithmetic 1e-5 relative
Frobenius, as everywhere for that arithmetic.
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


def _rank_k(u, s, v):
    return (u.double().cpu().numpy() * s.double().cpu().numpy()) @ v.double().cpu().numpy().T


@pytest.mark.parametrize("n,m,k,l,p", [
    (4225, 257, 8, 65, 4),     # one column past a 64-wide tile, odd K
    (5000, 300, 20, 130, 3),   # ragged rows, blocks and tiles
    (4096, 256, 16, 64, 1),    # exact tiles
    (33000, 129, 12, 128, 8),  # long Grams: K split over many launches
    (6000, 2048, 10, 90, 5),   # K over many folds
])
def test_rsvd_f64_matches_oracle(lib, n, m, k, l, p):
    a, _ = synth.haar_spectrum(n, m, seed=7 + n)
    u, s, v = lib.bsrht_rsvd(torch.from_numpy(a).cuda(), k, l, p, 3)
    ur, sr, vr = orc.rsvd(a, k, l, p, 3)
    assert np.max(np.abs(s.cpu().numpy() - sr)) <= 1e-12 * sr[0]
    ref = (ur * sr) @ vr.T
    assert np.linalg.norm(_rank_k(u, s, v) - ref) <= 1e-12 * np.linalg.norm(ref)


def test_rsvd_f64_column_scales(lib):
    """Rows and columns 2^-30 .. 2^30 apart keep the normwise accuracy."""
    a, _ = synth.haar_spectrum(4500, 200, seed=11)
    rng = np.random.default_rng(5)
    a = a * np.exp2(rng.integers(-30, 31, size=(4500, 1))) * np.exp2(rng.integers(-6, 7, size=(1, 200)))
    u, s, v = lib.bsrht_rsvd(torch.from_numpy(a).cuda(), 8, 80, 4, 3)
    ur, sr, vr = orc.rsvd(a, 8, 80, 4, 3)
    ref = (ur * sr) @ vr.T
    assert np.linalg.norm(_rank_k(u, s, v) - ref) <= 1e-12 * np.linalg.norm(ref)


def test_smaller_workspace_still_runs(lib):
    """A workspace short of the reported size takes the forms that fit."""
    n, m, k, l, p = 8192, 256, 16, 96, 4
    a, _ = synth.haar_spectrum(n, m, seed=12)
    x = torch.from_numpy(a).cuda()
    need = lib.bsrht_rsvd_workspace(n, m, k, l, p, torch.float64)
    ref = _rank_k(*lib.bsrht_rsvd(x, k, l, p, 9))
    for less in (256, 8 << 20):
        ws = torch.empty(need - less, device="cuda", dtype=torch.uint8)
        got = _rank_k(*lib.bsrht_rsvd(x, k, l, p, 9, workspace=ws))
        assert np.linalg.norm(got - ref) <= 1e-12 * np.linalg.norm(ref)
    with pytest.raises(lib.BsrhtError) as e:
        lib.bsrht_rsvd(x, k, l, p, 9, workspace=torch.empty(1 << 20, device="cuda", dtype=torch.uint8))
    assert e.value.status == -12


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float16])
@pytest.mark.parametrize("n,m,ld,l", [
    (1000, 208, 208, 17),   # narrow tile, ragged rows
    (4097, 200, 256, 64),   # column slice of a wider matrix
    (2048, 520, 520, 272),  # two column tiles of 144, K past a block of 64
    (2048, 264, 264, 256),  # one full 256-wide tile
    (1030, 203, 203, 40),   # rows off 16 bytes: the CUDA-core product
])
def test_rsvd_16bit_matches_oracle(lib, dtype, n, m, ld, l):
    a, _ = synth.haar_spectrum(n, m, seed=n + m, decay=20.0)
    buf = torch.zeros(n, ld, dtype=dtype)
    buf[:, :m] = torch.from_numpy(a).to(dtype)
    x = buf.cuda()[:, :m]
    u, s, v = lib.bsrht_rsvd(x, 10, l, 4, 5)
    vals = x.double().cpu().numpy()
    ur, sr, vr = orc.rsvd(vals, 10, l, 4, 5)
    ref = (ur * sr) @ vr.T
    assert np.max(np.abs(s.cpu().numpy() - sr)) <= 1e-5 * sr[0]
    assert np.linalg.norm(_rank_k(u, s, v) - ref) <= 1e-5 * np.linalg.norm(ref)


@pytest.mark.parametrize("n,m,ld,l", [
    (12300, 1028, 1028, 130),  # ragged rows, two column tiles, ragged last K block
    (12288, 1024, 1024, 128),  # one narrow tile: the TF32 product
    (12290, 2000, 2048, 257),  # column slice, little more than a wave: the TF32 product
    (16384, 1024, 1024, 256),  # exact tiles
    (16500, 1100, 1104, 257),  # column slice, one column past a tile, odd number of row tiles
    (12290, 1026, 1026, 130),  # rows off 16 bytes: the TF32 product
])
def test_rsvd_f32_matches_oracle(lib, n, m, ld, l):
    a, _ = synth.haar_spectrum(n, m, seed=n + m, decay=20.0)
    rng = np.random.default_rng(l)
    buf = torch.zeros(n, ld)
    # Rows 2^-40 .. 1 apart: each is split under its own scale.
    buf[:, :m] = torch.from_numpy(a * np.exp2(rng.integers(-40, 1, size=(n, 1))))
    x = buf.cuda()[:, :m]
    u, s, v = lib.bsrht_rsvd(x, 10, l, 4, 5)
    ur, sr, vr = orc.rsvd(x.double().cpu().numpy(), 10, l, 4, 5)
    ref = (ur * sr) @ vr.T
    assert np.max(np.abs(s.cpu().numpy() - sr)) <= 1e-5 * sr[0]
    assert np.linalg.norm(_rank_k(u, s, v) - ref) <= 1e-5 * np.linalg.norm(ref)
