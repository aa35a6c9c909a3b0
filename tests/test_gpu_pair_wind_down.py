"""Short products on CTA pairs back to back: each starts on SMs that a pair has just left, and every repetition gives the
same bits (residue products from N = 700, the 16-bit products of a factorization from about N = 2300)."""
import numpy as np
import pytest

from paper_2404_19163_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [705, 1024])
def test_repeated_residuals(n):
    import torch
    from paper_2404_19163_gb300 import Context, build
    build.build()
    S = synth.gaussian_overlap_torch(synth.cubic_sites(11, 2.5, 0.1, 1)[:n])
    Z = torch.eye(n, dtype=torch.float64, device="cuda") - 0.5 * (S - torch.eye(n, dtype=torch.float64, device="cuda"))
    exact = torch.eye(n, dtype=torch.float64, device="cuda") - Z.T @ (S @ Z)
    with Context(0) as c:
        first = torch.empty_like(S)
        err = c.residual(S, Z, "ozaki", D=first)
        # FP64 sums of N terms of |Z|^T|S||Z| < 16 err by a few N 2^-53 of it
        assert float((first - exact).abs().max()) <= 64.0 * n * 2.0 ** -53
        for _ in range(40):
            D = torch.empty_like(S)
            assert c.residual(S, Z, "ozaki", D=D) == err and torch.equal(D, first)


def test_repeated_factorizations():
    import torch
    from paper_2404_19163_gb300 import Context, build
    build.build()
    S = synth.gaussian_overlap_torch(synth.cubic_sites(14, 2.5, 0.1, 2)[:2601])
    with Context(0) as c:
        first = c.refine(S, None, order=2, precision="bf16_split", tol=1e-12)
        for _ in range(10):
            r = c.refine(S, None, order=2, precision="bf16_split", tol=1e-12)
            assert torch.equal(r.Z, first.Z) and np.array_equal(r.hist, first.hist)
