"""SVD of the l x l core at the edges of its forms: one CTA up to l = 64, a
cluster with columns of 64 to 768, the general sweeps beyond; 16-wide blocks of
the Cholesky; 32-wide tiles of small FP64 products.

Tolerances as for the whole calls: FP64 parity 1e-12, FP32 arithmetic 1e-5.
"""

import numpy as np
import pytest
import torch

import synth
from oracle import lowrank as orc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("l,k", [(16, 16), (33, 5), (64, 10), (65, 65), (128, 20), (129, 129), (256, 256), (257, 30),
                                 (512, 40), (513, 513), (768, 20), (769, 20)])
def test_core_svd_edges(dtype, l, k):
    import paper_2210_11295_gb300 as lib

    m = max(70, l + 3)
    n = 4 * m
    a, _ = synth.haar_spectrum(n, m, seed=l, decay=60.0)
    x = torch.from_numpy(a).to(dtype)
    u, s, v = lib.bsrht_rsvd(x.cuda(), k, l, 3, 11)
    ur, sr, vr = orc.rsvd(x.double().numpy(), k, l, 3, 11)
    tol = 1e-12 if dtype is torch.float64 else 1e-5
    u, s, v = (t.double().cpu().numpy() for t in (u, s, v))
    ref = (ur * sr) @ vr.T
    assert np.max(np.abs(s - sr)) <= tol * sr[0]
    assert np.linalg.norm((u * s) @ v.T - ref) <= tol * np.linalg.norm(ref)
