"""The FP64 path's products by CRT residues (N >= 320) against the same path on the CUDA cores (the slices setting
keeps it there) and against the FP64 oracle."""
import math

import numpy as np
import pytest

import oracle
from paper_2404_19163_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_2404_19163_gb300 import Context, build
    build.build()
    c = Context(0)
    yield c
    c.close()


def dev(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def both(ctx, S, Z0=None, **kw):
    out = []
    for scheme in ("auto", "slices"):
        ctx.set_emulation(scheme)
        out.append(ctx.refine(S, Z0, precision="fp64", **kw))
    ctx.set_emulation("auto")
    return out


def close(a, b, n, cond):
    """Two FP64-accurate factors: sums of N terms differ by a few sqrt(N) 2^-53 of |Z| a product, times cond(S)
    through the last update's residual; the history's entries at the floor by N 2^-53 per unit of |Z|^T|S||Z|."""
    za, zb = (x.Z.cpu().numpy() if hasattr(x.Z, "cpu") else x.Z for x in (a, b))
    assert np.linalg.norm(za - zb) <= 16.0 * math.sqrt(n) * cond * 2.0 ** -53 * np.linalg.norm(zb)
    m = min(len(a.hist), len(b.hist))
    assert np.allclose(a.hist[:m], b.hist[:m], rtol=1e-9, atol=16.0 * n * cond * 2.0 ** -53)


@pytest.mark.parametrize("n,order", [(319, 2), (320, 2), (321, 3), (383, 4), (449, 5), (513, 2)])
def test_cold(ctx, n, order):
    S, Q, lam = synth.householder_spd(n, seed=n)
    a, b = both(ctx, dev(S), order=order, fixed_iters=5)
    close(a, b, n, 25.0)
    Zo, ho, it = oracle.refine(S, None, m=order, nmax=50, fixed_iters=5)
    assert np.linalg.norm(a.Z.cpu().numpy() - Zo) <= 1e-12 * np.linalg.norm(Zo)
    assert a.info["iters"] == 5 and len(a.hist) == 6


def test_residual_at_the_floor_is_no_larger(ctx):
    """A decaying overlap, whose far entries an FP64 sum keeps to their own precision."""
    S = dev(synth.cubic_overlap(n_side=8))
    a, b = both(ctx, S, order=2)
    assert a.info["iters"] == b.info["iters"] and a.info["resid_f"] <= b.info["resid_f"]


def test_warm_host_and_unsymmetric_start(ctx):
    n = 333
    S, Q, lam = synth.householder_spd(n, seed=2)
    Z0 = (Q * lam ** -0.5) @ Q.T + 1e-3 * np.random.default_rng(5).standard_normal((n, n))
    a, b = both(ctx, np.ascontiguousarray(S), np.ascontiguousarray(Z0), order=2, fixed_iters=3)
    close(a, b, n, 25.0)


def test_graded_overlap(ctx):
    """Scales over four decades: Z's largest entry asks for more bits a row (past 62), then for more than the
    moduli hold, where the products go back to the CUDA cores."""
    n = 330
    S, Q, lam = synth.householder_spd(n, seed=4)
    for decades in (2.0, 5.0):
        d = 10.0 ** np.linspace(-decades, 0.0, n)
        Sg = dev(d[:, None] * S * d[None, :])
        Zs = dev((Q * lam ** -0.5) @ Q.T / d[:, None] * (1.0 + 1e-4))
        a, b = both(ctx, Sg, Zs, order=2, fixed_iters=2)
        za, zb = a.Z * dev(d)[:, None], b.Z * dev(d)[:, None]
        assert float((za - zb).norm() / zb.norm()) <= 1e-10
        assert abs(a.hist[0] - b.hist[0]) <= 1e-9 * b.hist[0]


def test_nonfinite_and_workspace_limit(ctx):
    from paper_2404_19163_gb300 import Context, ZfactError
    n = 400
    S, Q, lam = synth.householder_spd(n, seed=6)
    for where in ((3, 9), (7, 7)):
        Sn = S.copy()
        Sn[where] = Sn[where[::-1]] = np.nan
        with pytest.raises(ZfactError) as e:
            ctx.refine(dev(Sn), None, order=2, precision="fp64")
        assert e.value.code == 4
    # under a workspace cap: the CUDA-core path, with its bits and within its buffers
    with Context(0) as c2:
        c2.set_workspace_limit(6 * 8 * n * n + (1 << 20))
        r = c2.refine(dev(S), None, order=2, precision="fp64")
        ctx.set_emulation("slices")
        want = ctx.refine(dev(S), None, order=2, precision="fp64")
        ctx.set_emulation("auto")
        assert np.array_equal(r.Z.cpu().numpy(), want.Z.cpu().numpy())
        c2.set_workspace_limit(0)
