"""The sketch of FP32 and 16-bit rows off 16 bytes (row copies into the same
ring as the tensor maps): offsets of the base and of the stride, ragged
blocks and panels, the last rows of the matrix, every sketch-row group.

Tolerance: 1e-5 relative Frobenius against the FP64 oracle on the same
values, as everywhere for FP32 arithmetic.
"""

import numpy as np
import pytest
import torch

import synth
from oracle import bsrht as orc

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib():
    import paper_2210_11295_gb300 as m

    m.bsrht_sketch_autotune_reset()
    return m


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16, torch.float16])
@pytest.mark.parametrize("n,m,ld,off,p,l", [
    (2048, 33, 33, 0, 1, 64),      # one column past a panel, odd stride
    (2048, 33, 33, 1, 4, 64),      # base one element off as well
    (5003, 101, 103, 0, 3, 300),   # ragged blocks, columns of a wider matrix
    (1537, 7, 7, 3, 2, 200),       # windows wider than a row: many rows at the end
    (4096, 64, 66, 2, 2, 520),     # sketch-row groups of 1024, l just past 512
    (9001, 250, 250, 1, 6, 1024),  # the largest group, 2-byte and 4-byte offsets
    (20000, 97, 97, 0, 8, 1100),   # two groups
    (3000, 64, 64, 1, 4, 100),     # aligned stride, base off
])
def test_rows_off_16_bytes(lib, dtype, n, m, ld, off, p, l):
    base = synth.gaussian(n, ld, seed=n + m + off)
    flat = torch.full((n * ld + off,), float("nan"), dtype=dtype)
    flat[off:] = torch.from_numpy(base).to(dtype).reshape(-1)
    # Only the matrix itself lies in the buffer: its last row ends at its end.
    flat = flat[: off + (n - 1) * ld + m].clone().cuda()
    a = flat.as_strided((n, m), (ld, 1), off)
    b = lib.bsrht_sketch(a, p, l, 11)
    vals = a.double().cpu().numpy()
    ref = orc.sketch_fast(vals, p, l, 11)
    got = b.double().cpu().numpy()
    assert np.linalg.norm(got - ref) <= 1e-5 * np.linalg.norm(ref)
    again = lib.bsrht_sketch(a, p, l, 11)
    assert torch.equal(b, again)
