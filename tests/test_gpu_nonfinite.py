"""Matrices with a NaN or an Inf: a call returns (with an error status or not)
and leaves the library as it was.  The ranks of NaN norms must be a permutation,
which the kernels that gather by rank read as indices.
"""

import pytest
import torch

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib():
    import paper_2210_11295_gb300 as m

    return m


def _returns(lib, call):
    try:
        call()
    except lib.BsrhtError:
        pass
    torch.cuda.synchronize()


@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
@pytest.mark.parametrize("dtype,l", [
    (torch.float64, 40),    # one CTA's Jacobi
    (torch.float64, 100),   # cluster form
    (torch.float64, 800),   # sweeps beyond it
    (torch.float32, 100),
    (torch.float32, 800),
    (torch.bfloat16, 100),
])
def test_rsvd_nonfinite(lib, dtype, l, bad):
    n, m = 2048, max(200, l + 8)
    good = torch.from_numpy(synth.haar_spectrum(n, m, seed=l, decay=60.0)[0]).to(dtype).cuda()
    before = lib.bsrht_rsvd(good, 20, l, 4, 1)
    a = good.clone()
    a[77, 5] = bad
    _returns(lib, lambda: lib.bsrht_rsvd(a, 20, l, 4, 1))
    if dtype is not torch.bfloat16:
        _returns(lib, lambda: lib.bsrht_srsvd(a, 10, min(l, 90), min(l + 20, 180), 4, 1))
    after = lib.bsrht_rsvd(good, 20, l, 4, 1)
    assert all(torch.equal(x, y) for x, y in zip(before, after))


@pytest.mark.parametrize("dtype,precision", [(torch.float64, 0), (torch.float32, 0), (torch.float32, 1)])
@pytest.mark.parametrize("l", [40, 100])
def test_nystrom_nonfinite(lib, dtype, precision, l):
    good = torch.from_numpy(synth.psd_lowrank(2048, 150, seed=l)).to(dtype).cuda()
    before = lib.bsrht_nystrom(good, 20, l, 4, 1, precision=precision)
    a = good.clone()
    a[5, 5] = float("nan")
    _returns(lib, lambda: lib.bsrht_nystrom(a, 20, l, 4, 1, precision=precision))
    after = lib.bsrht_nystrom(good, 20, l, 4, 1, precision=precision)
    assert all(torch.equal(x, y) for x, y in zip(before, after))
