"""The FP64 precision holds every entry of the factor to FP64 arithmetic's own error, the far entries of a decaying
overlap among them: a product's entry errs by at most N 2^-53 of (|A||B|)_ij (plus the storing of A and B), and an update
Z (I + Q(d)) chains four of them, so |Z - Z_exact|_ij <= 8 N 2^-53 (|Z| (I + M/2 + 3/8 M^2))_ij with
M = I + |Z|^T |S| |Z|; the same for the oracle's Z."""
import numpy as np
import pytest

import oracle
from paper_2404_19163_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("side,n", [(6, 200), (7, 320), (7, 343), (9, 601)])
def test_far_entries(side, n):
    import torch
    from paper_2404_19163_gb300 import Context, build
    build.build()
    S = np.ascontiguousarray(synth.cubic_overlap(n_side=side)[:n, :n])
    with Context(0) as c:
        r = c.refine(torch.from_numpy(S).cuda(), None, order=2, precision="fp64")
        Zf = c.refine(torch.from_numpy(S).cuda(), None, order=2, precision="fp64", fixed_iters=4).Z.cpu().numpy()
    Zo, _, _ = oracle.refine(S, None, m=2, nmax=50, fixed_iters=4)
    a = np.abs(Zo)
    M = np.eye(n) + a.T @ (np.abs(S) @ a)
    W = a @ (np.eye(n) + M / 2 + 3.0 / 8.0 * M @ M)
    assert a.min() < 1e-17 * a.max()
    for Z in (r.Z.cpu().numpy(), Zf):
        assert np.all(np.abs(Z - Zo) <= 16.0 * n * 2.0 ** -53 * W)
