"""FP32 products at the edges of their tiles."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_2404_19163_gb300 import Context, build
    build.build()
    c = Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("n", [1, 3, 63, 64, 65, 130, 319, 384, 449, 2047, 2049])
def test_f32_tiles(ctx, n):
    import torch
    g = torch.Generator(device="cuda").manual_seed(n)
    A, B = (torch.randn((n, n), dtype=torch.float64, device="cuda", generator=g) for _ in range(2))
    C = ctx.gemm(A, B, precision="fp32")
    A32, B32 = A.float().double(), B.float().double()
    # a chain of n FP32 FMAs errs by at most n 2^-24 of the sum of magnitudes
    assert bool(((C - A32 @ B32).abs() <= 1.01 * n * 2.0 ** -24 * (A32.abs() @ B32.abs())).all())
    # d = I - X through the factorization's symmetric tiles: mirrored exactly
    S = torch.eye(n, dtype=torch.float64, device="cuda") + 0.1 * (A @ A.T) / n
    r = ctx.refine(S, None, order=3, precision="fp32", fixed_iters=6)
    assert r.info["resid_f"] / n ** 0.5 <= 1e-5
