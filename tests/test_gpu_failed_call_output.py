"""A factorization that fails before its result is known leaves a device Z alone, and with it a start that Z aliases."""
import numpy as np
import pytest

from paper_2404_19163_gb300 import synth

pytestmark = pytest.mark.gpu

NOMEM = 3


@pytest.mark.parametrize("n,steps", [(48, -1), (300, -1), (300, 2), (700, -1)])
@pytest.mark.parametrize("warm", [False, True])
def test_workspace_refusals_leave_z_alone(n, steps, warm):
    import torch
    from paper_2404_19163_gb300 import Context, build
    build.build()
    side = int(np.ceil(n ** (1.0 / 3.0)))
    S = synth.gaussian_overlap_torch(synth.cubic_sites(side, 2.5, 0.1, 1)[:n])
    start = torch.eye(n, dtype=torch.float64, device="cuda") * 0.9

    def status(cap):
        Z = start.clone()  # Z aliases the start of a warm call
        with Context(0) as c:
            c.set_workspace_limit(cap)
            r = c.refine(S, Z if warm else None, order=2, precision="bf16", Z=Z, refine_steps=steps, tol=0.0,
                         raise_on_error=False)
        assert r.status != NOMEM or torch.equal(Z, start), cap
        return r.status

    lo, hi = 0, 1 << 34
    while hi - lo > 256:  # the least cap that holds the call, and every refusal on the way
        mid = (lo + hi) // 2
        lo, hi = (mid, hi) if status(mid) == NOMEM else (lo, mid)
    for cap in np.linspace(0.5 * lo, lo, 24):
        assert status(int(cap)) == NOMEM
