"""Odd sizes over workspace that holds stale NaN patterns: what lies past an operand's last row stays out of the
residue products' results (single and grouped calls)."""
import numpy as np
import pytest

import oracle
from paper_2404_19163_gb300 import synth

pytestmark = pytest.mark.gpu


def stale():
    import torch
    torch.cuda.empty_cache()
    x = torch.full((1 << 28,), float("nan"), dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    del x
    torch.cuda.empty_cache()


def test_residual_and_batched():
    import torch
    from paper_2404_19163_gb300 import Context, build
    build.build()
    sizes = [65, 131, 97, 33]
    S = [synth.householder_spd(n, seed=n)[0] for n in sizes]
    dev = [torch.from_numpy(s).cuda() for s in S]
    stale()
    with Context(0) as c:
        Z, hist, infos, status = c.refine_batched(dev, None, [2] * len(S), precision="bf16_split")
        for s, z, i in zip(S, Z, infos):
            _, e = oracle.residual(s, z.cpu().numpy())
            assert abs(i["resid_f"] - e) <= 1e-12 * max(1.0, e) + 1e-9 * e
    stale()
    with Context(0) as c:
        for s, d, z in zip(S, dev, Z):
            D, e = oracle.residual(s, z.cpu().numpy())
            out = torch.empty_like(d)
            assert abs(c.residual(d, z, "ozaki", D=out) - e) <= 1e-12 * max(1.0, e) + 1e-9 * e
            assert np.max(np.abs(out.cpu().numpy() - D)) <= 1e-12
