"""The bulk that the host queues ahead of the device's decisions (graphs on) against the host loop: short limits, starts
that are not finite, outputs over inputs.  Status, counts, history and result are the same."""
import numpy as np
import pytest

from paper_2404_19163_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_2404_19163_gb300 import Context, build
    build.build()
    c = Context(0)
    yield c
    c.close()


CASES = {
    "cold": {}, "cold_nmax1": {"nmax": 1}, "cold_nmax2": {"nmax": 2}, "warm": {}, "warm_nmax1": {"nmax": 1},
    "cold_nan": {}, "warm_nan_s": {}, "warm_nan_z": {}, "cold_rule1": {"stop_rule": 1, "tol": 1e-3},
    "out_is_start": {}, "out_is_s": {}, "no_refinement": {"refine_steps": 0}, "fp32_refinement": {"refine_mode": 2},
    "start_scale": {"start_scale": 2.0},
}


@pytest.mark.parametrize("precision", ["bf16_split", "fp16_split", "fp16"])
@pytest.mark.parametrize("what", sorted(CASES))
def test_same_as_the_host_loop(ctx, what, precision):
    import torch
    n = 201
    S, Q, lam = synth.householder_spd(n, seed=31)
    start = (Q * lam ** -0.5) @ Q.T + 2e-3 * np.random.default_rng(1).standard_normal((n, n))
    if what in ("cold_nan", "warm_nan_s"):
        S[4, 7] = S[7, 4] = np.nan
    if what == "warm_nan_z":
        start[5, 2] = np.nan
    out = []
    for graphs in (True, True, False):  # the graph's first use and a later one
        ctx.set_loop_graphs(graphs)
        Sd = torch.from_numpy(S.copy()).cuda()
        Z0 = torch.from_numpy(start.copy()).cuda() if what.startswith("warm") or what == "out_is_start" else None
        Z = {"out_is_start": Z0, "out_is_s": Sd}.get(what)
        out.append(ctx.refine(Sd, Z0, order=3, precision=precision, Z=Z, raise_on_error=False, **CASES[what]))
    ctx.set_loop_graphs(True)
    for a in out[:2]:
        b = out[2]
        assert a.status == b.status
        assert a.info["iters"] == b.info["iters"] and a.info["refine_iters"] == b.info["refine_iters"]
        assert np.array_equal(a.hist, b.hist, equal_nan=True)
        assert np.array_equal(a.Z.cpu().numpy(), b.Z.cpu().numpy(), equal_nan=True)
    if "nan" in what:
        assert out[0].status == 4 and out[0].info["iters"] == 0 and len(out[0].hist) == 1
