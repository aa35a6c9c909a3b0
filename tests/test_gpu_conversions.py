"""FP64 values to 16-bit operands at the ends of FP32's range and of the conversion kernels' tiles: rows (the left
operand of a product with the identity) and columns (the right one), against torch's conversions."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_2404_19163_gb300 import Context, build
    build.build()
    c = Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("n", [1, 2, 3, 31, 32, 33, 63, 64, 65, 130])
@pytest.mark.parametrize("scale", [1.0, 2.0 ** -20, 2.0 ** 12, 1.5])
def test_bf16_hi_lo(ctx, n, scale):
    import torch
    g = np.random.default_rng(n)
    a = g.standard_normal((n, n)) * 2.0 ** g.integers(-160, 60, (n, n))
    edge = np.array([0.0, -0.0, 2.0 ** -126, 2.0 ** -149, 2.0 ** -150, 1.5 * 2.0 ** -150, -(2.0 ** -151), 1e-300, 5e-324,
                     1.0 + 2.0 ** -24, 1.0 + 3 * 2.0 ** -24, 1.0 + 2.0 ** -24 + 2.0 ** -52, 2.0 - 2.0 ** -25])
    a.ravel()[:edge.size] = edge[:a.size]
    A = torch.from_numpy(a).cuda()
    eye = torch.eye(n, dtype=torch.float64, device="cuda")
    x = (A * scale).float()
    hi = x.bfloat16().float()
    want = hi + (x - hi).bfloat16().float()  # exact in FP32, and the product's sum
    want = torch.where(want.abs() < 2.0 ** -110, torch.zeros_like(want), want).double() / scale
    for C in (ctx.gemm(A, eye, precision="bf16_split", scale_a=scale), ctx.gemm(eye, A, precision="bf16_split", scale_b=scale)):
        C = torch.where(C.abs() * scale < 2.0 ** -110, torch.zeros_like(C), C)  # (the tensor cores may flush subnormals)
        # the epilogue divides by FP32(scale)
        assert bool(((C - want).abs() <= 2.0 ** -23 * want.abs()).all()) if scale == 1.5 else torch.equal(C, want)
