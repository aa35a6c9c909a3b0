"""Workspace caps that hold a call: the least ones of an earlier build, whose statistics took one scratch row per column and
whose moduli came from measured norms at every size.  A capped call takes the measured norms and gives the uncapped bits."""
import numpy as np
import pytest

from paper_2404_19163_gb300 import learn, synth

pytestmark = pytest.mark.gpu

CAPS = {
    "bf16": {64: 2719040, 300: 33082432, 1000: 264668672, 1500: 595429952, 2100: 1199848896},
    "bf16_split": {64: 2735424, 300: 33691712, 1000: 266323456, 1500: 599153216, 2100: 1221289920},
    "fp16_split.warm": {64: 2653504, 300: 32652352, 1000: 258033152, 1500: 589937216, 2100: 1184084928},
    "bf16.m4": {64: 2866496, 300: 35705792, 1000: 290174976, 1500: 664560320, 2100: 1336150080},
    "bf16.bulk": {64: 181312, 300: 4129600, 1000: 44677120, 1500: 100522240, 2100: 194765120},
    "fp16_split.bulk": {64: 246848, 300: 5665600, 1000: 61061120, 1500: 137386240, 2100: 265728320},
    "bf16.resid": {64: 1865024, 300: 23897792, 1000: 195479808, 1500: 439779008, 2100: 879484224},
    "steps2": {64: 2719040, 300: 33082432, 1000: 264668672, 1500: 595429952, 2100: 1199848896},
    "fp32.refine": {64: 1971584, 300: 26066432, 1000: 219492224, 1500: 493789568, 2100: 985333632},
    "fp32.ozaki": {64: 2513216, 300: 29940032, 1000: 236984448, 1500: 533124352, 2100: 1075301824},
    "residual": {64: 1634560, 300: 18664192, 1000: 138706688, 1500: 312040768, 2100: 631698304},
    "residual.slices": {64: 1167616, 300: 15205632, 1000: 125583104, 1500: 365456704, 2100: 723494272},
    "congruence": {64: 1571840, 300: 17999040, 1000: 125095296, 1500: 281428416, 2100: 573484608},
    "batched": {64: 8615744, 300: 85910272, 1000: 549576256, 1500: 1236462016, 2100: 2550107392},
    "batched.steps": {64: 3784960, 300: 40751872, 1000: 285058816, 1500: 641306432, 2100: 1327126016},
    "propose": {64: 84736, 300: 1843264, 1000: 20153536, 1500: 45285568, 2100: 88384768},
}


def cubic(n, seed=0):
    side = int(np.ceil(round(n ** (1.0 / 3.0), 9)))
    return synth.gaussian_overlap_torch(synth.cubic_sites(side, 2.5, 0.1, seed)[:n])


def refine(c, S, Z0, precision, **kw):
    r = c.refine(S, Z0, order=kw.pop("order", 2), precision=precision, **kw)
    return [r.Z, r.hist, r.info["iters"], r.info["refine_iters"]]


def residual(c, S, Z0):
    return [c.residual(S, Z0, "ozaki")]


def slices(c, S, Z0):
    c.set_emulation("slices")
    return residual(c, S, Z0)


def batched(c, S, **kw):
    Z, hist, infos, status = c.refine_batched([S, S], None, [2, 2], precision="bf16_split", **kw)
    return [Z[0], Z[1]] + [i["resid_f"] for i in infos]


CALLS = {
    "bf16": lambda c, S, Z0: refine(c, S, None, "bf16"),
    "bf16_split": lambda c, S, Z0: refine(c, S, None, "bf16_split", tol=1e-12),
    "fp16_split.warm": lambda c, S, Z0: refine(c, S, Z0, "fp16_split", tol=1e-12),
    "bf16.m4": lambda c, S, Z0: refine(c, S, None, "bf16", order=4),
    "bf16.bulk": lambda c, S, Z0: refine(c, S, None, "bf16", refine_steps=0, final_residual=0),
    "fp16_split.bulk": lambda c, S, Z0: refine(c, S, None, "fp16_split", refine_steps=0, final_residual=0),
    "bf16.resid": lambda c, S, Z0: refine(c, S, None, "bf16", refine_steps=0),
    "steps2": lambda c, S, Z0: refine(c, S, None, "bf16", refine_steps=2, tol=0.0),
    "fp32.refine": lambda c, S, Z0: refine(c, S, None, "bf16", refine_mode="fp32"),
    "fp32.ozaki": lambda c, S, Z0: refine(c, S, None, "fp32", refine_steps=1),
    "residual": residual,
    "residual.slices": slices,
    "congruence": lambda c, S, Z0: [c.congruence(S * 0.5, Z0)],
    "batched": lambda c, S, Z0: batched(c, S),
    "batched.steps": lambda c, S, Z0: batched(c, S, refine_steps=1),
    "propose": lambda c, S, Z0: list(c.propose(S, *learn.load()[:3])),
}


@pytest.mark.parametrize("n", [64, 300, 1000, 1500, 2100])
@pytest.mark.parametrize("call", list(CAPS))
def test_cap_still_holds_the_call(call, n):
    import torch
    from paper_2404_19163_gb300 import Context, build
    build.build()
    S = cubic(n)
    with Context(0) as c:
        Z0 = c.refine(cubic(n, 3), None, order=2, precision="bf16_split").Z
    out = []
    for cap in (0, CAPS[call][n]):
        with Context(0) as c:
            c.set_workspace_limit(cap)
            out.append(CALLS[call](c, S, Z0))
    for a, b in zip(*out):
        assert torch.equal(a, b) if torch.is_tensor(a) else np.array_equal(a, b)
