"""Symmetric residue products of more than 20 moduli over workspace whose bytes are all 255: the digits below the
diagonal, which no product writes, neither index the reconstruction's table nor reach the result."""
import numpy as np
import pytest

import oracle
from paper_2404_19163_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [130, 401, 1001, 1530, 2050])
def test_residual_over_bytes_of_255(n):
    import torch
    from paper_2404_19163_gb300 import Context, build
    build.build()
    side = int(np.ceil(n ** (1.0 / 3.0)))
    S = synth.cubic_overlap(n_side=side)[:n, :n].copy()
    # max|Z|^2 g_hi between 2^19 and 2^25 asks for 78 bits a row, 21 moduli and more
    Z = 1024.0 * (np.eye(n) + 1e-3 * np.random.default_rng(n).standard_normal((n, n)))
    assert 2.0 ** 19 < np.max(np.abs(Z)) ** 2 * np.max(np.abs(S).sum(axis=1)) < 2.0 ** 25
    d_or, err_or = oracle.residual(S, Z)
    Sd, Zd = torch.from_numpy(S).cuda(), torch.from_numpy(Z).cuda()
    D = torch.empty_like(Sd)
    torch.cuda.empty_cache()
    x = torch.full((1 << 31,), 255, dtype=torch.uint8, device="cuda")
    torch.cuda.synchronize()
    del x
    torch.cuda.empty_cache()
    with Context(0) as c:
        c.set_profiling(True)
        err = c.residual(Sd, Zd, "ozaki", D=D)
        stats = {k["name"]: k for k in c.kernel_stats()}
    assert "tc_gemm.ozaki" not in stats
    assert stats["tc_gemm.crt"]["flops"] >= 21 * (2.0 + 1.0) * n ** 3
    scale = float(np.max(np.abs(Z).T @ (np.abs(S) @ np.abs(Z))))
    assert np.max(np.abs(D.cpu().numpy() - d_or)) <= 1e-13 * scale
    assert abs(err - err_or) <= 1e-13 * scale * n
