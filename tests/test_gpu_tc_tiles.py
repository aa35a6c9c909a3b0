"""Every tile shape of the tensor-core engine at ragged sizes: the sizes span the choice of the shape (32-, 64-,
128-wide tiles of one CTA, 256 x 256 of a pair) and end inside a chunk, a tile and a pair.  A dense S (entries of
all blocks alike) makes a wrong block or mirror visible in every entry."""
import pytest

pytestmark = pytest.mark.gpu

U = {"bf16": 2.0 ** -8, "bf16_split": 2.0 ** -16, "fp16_split": 2.0 ** -20}


@pytest.fixture(scope="module")
def ctx():
    from paper_2404_19163_gb300 import Context, build
    build.build()
    c = Context(0)
    yield c
    c.close()


def _dense(n, seed):
    import torch
    g = torch.Generator(device="cuda").manual_seed(seed)
    E = torch.randn((n, n), dtype=torch.float64, device="cuda", generator=g) * (0.1 / n ** 0.5)
    S = E + E.T
    S.diagonal().add_(1.0)
    Z0 = torch.randn((n, n), dtype=torch.float64, device="cuda", generator=g) * (0.05 / n ** 0.5)
    Z0.diagonal().add_(1.0)
    return S, Z0


@pytest.mark.parametrize("prec,order", [("bf16_split", 2), ("fp16_split", 3), ("bf16", 2)])
@pytest.mark.parametrize("n", [31, 129, 333, 1000, 1187, 2309, 3700])
def test_one_update_elementwise(ctx, n, prec, order):
    import torch
    S, Z0 = _dense(n, n)
    Z = ctx.refine(S, Z0, order=order, precision=prec, fixed_iters=1, refine_steps=0, final_residual=0).Z
    d = torch.eye(n, dtype=torch.float64, device="cuda") - Z0.T @ (S @ Z0)
    P, Q, c = d, 0.5 * d, 0.5
    for k in range(2, order + 1):
        P, c = P @ d, c * (2 * k - 1) / (2 * k)
        Q = Q + c * P
    ref = Z0 + Z0 @ Q
    # operands rounded to the format (u), nseg K products summed in FP32 in any order: the relative errors of
    # d's two products (five roundings), the powers and the update act on |Z0| (1 + |Z0|^T |S| |Z0|)
    nseg = 3 if prec.endswith("split") else 1
    W = Z0.abs() + Z0.abs() @ (Z0.T.abs() @ (S.abs() @ Z0.abs()))
    bound = 6.0 * (3.0 * U[prec] + nseg * n * 2.0 ** -24) * W
    assert bool(((Z - ref).abs() <= bound).all()), float(((Z - ref).abs() / bound).max())


@pytest.mark.parametrize("n", [31, 333, 700, 1187, 2309])
def test_residual_entries(ctx, n):
    """The residue products' tiles: d to FP64 accuracy (relative to |Z|^T |S| |Z|) in every entry, symmetric."""
    import torch
    S, Z0 = _dense(n, 3 * n)
    D = torch.empty_like(S)
    ctx.residual(S, Z0, "ozaki", D=D)
    ref = torch.eye(n, dtype=torch.float64, device="cuda") - Z0.T @ (S @ Z0)
    ref = torch.triu(ref) + torch.triu(ref, 1).T
    assert torch.equal(D, D.T)
    assert float((D - ref).abs().max()) <= 1e-13 * float((Z0.T.abs() @ (S.abs() @ Z0.abs())).max())
