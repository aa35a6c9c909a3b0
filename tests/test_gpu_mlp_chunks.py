"""The start network's kernel at the edges of its 64-sample chunks."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_2404_19163_gb300 import Context, build
    build.build()
    c = Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("batch", [1, 2, 63, 64, 65, 130])
def test_mlp_chunks(ctx, batch):
    import torch
    g = np.random.default_rng(batch)
    f32 = lambda a: torch.from_numpy(np.asarray(a, dtype=np.float32)).cuda()  # noqa: E731
    P, x = 0.3 * g.standard_normal(oracle.mlp_num_params()), g.standard_normal((batch, 16))
    mean, std = 0.1 * g.standard_normal(16), g.uniform(0.5, 1.5, 16)
    ts, to = g.standard_normal(batch).astype(np.float32), g.integers(0, 4, batch).astype(np.int32)
    # parameters at an odd address, as a slice of a larger tensor has
    Pd = torch.cat([torch.zeros(1, device="cuda"), f32(P)])[1:]
    y = ctx.mlp_forward(Pd, f32(mean), f32(std), f32(x)).cpu().numpy()
    grad, loss = ctx.mlp_backward(Pd, f32(mean), f32(std), f32(x), f32(ts), torch.from_numpy(to).cuda(), 0.7)
    n32 = lambda a: np.asarray(a, dtype=np.float32)  # noqa: E731
    xn = ((n32(x) - n32(mean)) / n32(std)).astype(np.float64)
    P64 = n32(P).astype(np.float64)
    # FP32 sums of up to 64 terms through two layers, and of the batch
    assert np.allclose(y, oracle.mlp_forward(P64, xn), rtol=1e-4, atol=1e-4)
    want = oracle.mlp_backward(P64, xn, ts.astype(np.float64), to, 0.7)
    assert np.linalg.norm(grad.cpu().numpy() - want) <= 1e-4 * np.linalg.norm(want)
    lo = oracle.mlp_loss(P64, xn, ts.astype(np.float64), to, 0.7)
    assert abs(loss - lo) <= 1e-5 * abs(lo)
