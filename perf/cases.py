"""Performance cases: the calls a user of this library makes, over the sizes, precisions and starts in use.

Each case is a dict of plain values.  ``prepare`` makes what a program holds before the call (overlap matrices
built on the GPU from seeded geometries, a warm start, network weights; one library context per process, as a
program keeps one), ``run`` is one call through the public binding, ``exact`` the same result in plain torch in
64 bits.  The matrices are the library's own recipes (``synth``): jittered cubic Gaussian overlaps, random
clusters, multi-exponent fcc blocks, Householder SPD matrices and the paper's synthetic matrix.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2404_19163_gb300 import Context, learn, synth

_context = None


def context():
    global _context
    if _context is None:
        _context = Context(0)
    return _context


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # a small molecule: the bench's smallest workload, bound by latency
        {"name": "refine_n256", "op": "refine", "family": "householder", "n": 256, "precision": "bf16_split",
         "order": 2, "warm": False, "host": False, "tol": 1e-12},
        # the paper's synthetic matrix and perturbed start with the FP16 split (ragged: 1000 = 15.6 x 64)
        {"name": "refine_n1000_warm", "op": "refine", "family": "paper", "n": 1000, "precision": "fp16_split",
         "order": 2, "warm": True, "host": False, "tol": 1e-12},
        # a host program: pinned S in, pinned Z out, plain BF16 bulk of order 3 (13^3 sites, odd N)
        {"name": "refine_n2197_host", "op": "refine", "family": "cubic", "n": 2197, "precision": "bf16",
         "order": 3, "warm": False, "host": True, "tol": 1e-12},
        # the headline: one cold factorization of the N = 4096 cubic overlap to 1e-12
        {"name": "refine_n4096", "op": "refine", "family": "cubic", "n": 4096, "precision": "bf16_split",
         "order": 2, "warm": False, "host": False, "tol": 1e-12},
        # an ill-conditioned multi-exponent basis (cond ~ 7e5), warm-started from the previous geometry
        {"name": "refine_n8192_ill_warm", "op": "refine", "family": "fcc", "n": 8192, "precision": "fp16_split",
         "order": 2, "warm": True, "host": False, "tol": 1e-12},
        # the paper's "double": every product in FP64
        {"name": "refine_n729_fp64", "op": "refine", "family": "cubic", "n": 729, "precision": "fp64",
         "order": 2, "warm": False, "host": False, "tol": 0.0},
        # the paper's "single": every bulk product in FP32
        {"name": "refine_n1331_fp32", "op": "refine", "family": "cubic", "n": 1331, "precision": "fp32",
         "order": 2, "warm": False, "host": False, "tol": 0.0},
        # a frame of a trajectory of uneven clusters, warm-started from the previous frame, each with its
        # FP64-accurate residual
        {"name": "batched_32_clusters", "op": "batched", "count": 32, "lo": 256, "hi": 2048, "layout": 0,
         "precision": "bf16_split", "order": 2, "warm": True},
        # the consumer of Z: H_perp = Z^T H Z to FP64 accuracy
        {"name": "congruence_n3000", "op": "congruence", "n": 3000, "precision": "fp64", "mode": "ozaki"},
        # checking a Z that came from elsewhere: d = I - Z^T S Z and its norm to FP64 accuracy
        {"name": "residual_n1728", "op": "residual", "n": 1728, "mode": "ozaki"},
        # a learned start for a matrix not seen before: features and the network
        {"name": "propose_n1500", "op": "propose", "n": 1500},
        # one full-batch training step of the start network: gradients, then Adam
        {"name": "train_20000", "op": "train", "batch": 20000},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["refine"] * 5 + ["double", "single", "batched", "congruence", "residual", "propose", "train"])
    if op == "refine":
        family = rng.choice(["cubic", "cubic", "householder", "paper", "fcc"])
        hi = {"cubic": 4096, "householder": 512, "paper": 2048, "fcc": 6000}[family]
        return {"op": "refine", "family": family, "n": _log_int(rng, 96, hi),
                "precision": "fp16_split" if family == "fcc" else rng.choice(["bf16_split", "bf16_split", "fp16_split", "bf16"]),
                "order": 2 if family == "fcc" else rng.choice([2, 2, 2, 3, 4, 5]),
                "warm": family in ("paper", "fcc"), "host": rng.random() < 0.2, "tol": 1e-12}
    if op == "double":
        return {"op": "refine", "family": "cubic", "n": _log_int(rng, 64, 1024), "precision": "fp64",
                "order": rng.choice([2, 2, 3]), "warm": False, "host": False, "tol": 0.0}
    if op == "single":
        return {"op": "refine", "family": "cubic", "n": _log_int(rng, 64, 2500), "precision": "fp32",
                "order": rng.choice([2, 2, 3]), "warm": False, "host": False, "tol": 0.0}
    if op == "batched":
        lo = rng.randint(64, 512)
        return {"op": "batched", "count": rng.randint(3, 32), "lo": lo, "hi": lo + _log_int(rng, 64, 1536),
                "layout": rng.randint(1, 1 << 20), "precision": rng.choice(["bf16_split", "bf16_split", "bf16"]),
                "order": rng.choice([2, 2, 3]), "warm": rng.random() < 0.75}
    if op == "congruence":
        return {"op": "congruence", "n": _log_int(rng, 128, 4096), "precision": rng.choice(["fp64", "fp64", "bf16_split"]),
                "mode": "ozaki"}
    if op == "residual":
        mode = rng.choice(["ozaki", "ozaki", "native"])
        return {"op": "residual", "n": _log_int(rng, 64, 4096 if mode == "ozaki" else 1024), "mode": mode}
    if op == "propose":
        return {"op": "propose", "n": _log_int(rng, 128, 4096)}
    return {"op": "train", "batch": _log_int(rng, 256, 20000)}


# ------------------------------------------------------------------ inputs
def _cubic(n, seed):
    side = int(math.ceil(round(n ** (1.0 / 3.0), 9)))
    return synth.gaussian_overlap_torch(synth.cubic_sites(side, 2.5, 0.1, seed)[:n])


def _fcc(n, seed):
    # the smallest block of about cubic shape that holds n functions (16 per cell), cut at n
    cells = -(-n // 16)
    cx = max(1, int(round((cells / 2.0) ** (1.0 / 3.0))))
    cz = -(-cells // (cx * cx))
    pos = synth.fcc_sites((cx, cx, cz)) + synth.rng(3, 100 + seed).normal(0.0, 0.01, (4 * cx * cx * cz, 3))
    centres, a = synth.fcc_basis(pos)
    return synth.gaussian_overlap_torch(centres[:n], a[:n])


def _sizes(case):
    g = np.random.default_rng(case["layout"])
    return [int(v) for v in g.integers(case["lo"], case["hi"] + 1, case["count"])]


def _symmetric_normal(n, gen):
    B = torch.randn((n, n), dtype=torch.float64, device="cuda", generator=gen)
    return (B + B.T).mul_(0.5)


def prepare(case, seed):
    ctx, op = context(), case["op"]
    gen = torch.Generator(device="cuda").manual_seed(seed)
    s = {"case": case, "ctx": ctx}
    if op == "refine":
        n, Z0 = case["n"], None
        if case["family"] == "householder":
            S = torch.from_numpy(synth.householder_spd(n, seed)[0]).cuda()
        elif case["family"] == "paper":
            S = synth.paper_synthetic_torch(n)
            Z0 = synth.paper_start_torch(S, 0.005, seed)
        elif case["family"] == "fcc":
            S = _fcc(n, 2 * seed + 1)
            Z0 = ctx.refine(_fcc(n, 2 * seed), None, order=2, precision=case["precision"]).Z  # the previous geometry's
        else:
            S = _cubic(n, seed)
        Z = torch.empty_like(S)
        if case["host"]:
            S, Z = S.cpu().pin_memory(), Z.cpu().pin_memory()
            Z0 = Z0.cpu().pin_memory() if Z0 is not None else None
        s.update(S=S, Z0=Z0, Z=Z)
    elif op == "batched":
        sites = [synth.cluster_sites(n, (1000 * seed + i) % (1 << 31)) for i, n in enumerate(_sizes(case))]
        g, Z0 = np.random.default_rng(seed), None
        if case["warm"]:
            Z0 = ctx.refine_batched([synth.gaussian_overlap_torch(p) for p in sites], None, [case["order"]] * len(sites),
                                    precision=case["precision"])[0]
            sites = [p + g.normal(0.0, 0.02, p.shape) for p in sites]
        S = [synth.gaussian_overlap_torch(p) for p in sites]
        s.update(S=S, Z0=Z0, Z=[torch.empty_like(x) for x in S])
    elif op == "congruence":
        n = case["n"]
        Z = torch.randn((n, n), dtype=torch.float64, device="cuda", generator=gen).mul_(n ** -0.5)
        Z.diagonal().add_(1.0)
        s.update(H=_symmetric_normal(n, gen), Z=Z)
    elif op == "residual":
        n = case["n"]
        S = _cubic(n, seed)
        # the factor of a neighbouring geometry: (I - E/2 + 3E^2/8) of S = I + E, off by the series' tail
        E = S - torch.eye(n, dtype=torch.float64, device="cuda")
        Z = (E @ E).mul_(0.375).sub_(E, alpha=0.5)
        Z.diagonal().add_(1.0)
        s.update(S=S, Z=Z, D=torch.empty_like(S))
    elif op == "propose":
        P, mu, sd, _ = learn.load()
        s.update(S=_cubic(case["n"], seed), P=P, mu=mu, sd=sd)
    else:
        g, b = np.random.default_rng(seed), case["batch"]
        dev = lambda a, dt=torch.float32: torch.from_numpy(np.ascontiguousarray(a)).to("cuda", dt)  # noqa: E731
        p = learn.init_params(seed)
        s.update(X=dev(g.standard_normal((b, 16))), ts=dev(g.uniform(0.5, 1.5, b)), to=dev(g.integers(0, 4, b), torch.int32),
                 mu=dev(0.1 * g.standard_normal(16)), sd=dev(g.uniform(0.5, 1.5, 16)), P=dev(p),
                 # moments of a run that is under way
                 M=dev(1e-2 * g.standard_normal(p.size)), V=dev(g.uniform(1e-4, 4e-4, p.size)), step=100)
    return s


# ------------------------------------------------------------------ one pass
def run(s):
    case, ctx, op = s["case"], s["ctx"], s["case"]["op"]
    if op == "refine":
        r = ctx.refine(s["S"], s["Z0"], order=case["order"], precision=case["precision"], Z=s["Z"], tol=case["tol"])
        return {"Z": r.Z, "iters": r.info["iters"], "refine_iters": r.info["refine_iters"]}
    if op == "batched":
        Z, hist, infos, status = ctx.refine_batched(s["S"], s["Z0"], [case["order"]] * len(s["S"]),
                                                    precision=case["precision"], Z_list=s["Z"])
        return {"Z": Z, "resid": np.array([i["resid_f"] for i in infos]), "iters": np.array([i["iters"] for i in infos])}
    if op == "congruence":
        return {"Hp": ctx.congruence(s["H"], s["Z"], precision=case["precision"], mode=case["mode"])}
    if op == "residual":
        err = ctx.residual(s["S"], s["Z"], mode=case["mode"], D=s["D"])
        return {"D": s["D"], "err": np.array([err])}
    if op == "propose":
        scale, order = ctx.propose(s["S"], s["P"], s["mu"], s["sd"])
        return {"scale": np.array([scale]), "order": order}
    grad, loss = ctx.mlp_backward(s["P"], s["mu"], s["sd"], s["X"], s["ts"], s["to"])
    ctx.mlp_adam(s["P"], grad, s["M"], s["V"], s["step"])
    return {"grad": grad, "loss": np.array([loss]), "P": s["P"], "M": s["M"], "V": s["V"]}


# ------------------------------------------------------------------ what a pass cannot do without
# bulk updates of the method on these inputs (order 2), each 6 N^3 FLOPs: Z^T S, X, d^2 and Z Q
_UPDATES = {"householder": 6, "cubic": 3, "paper": 3, "fcc": 2}


def work(case):
    op = case["op"]
    if op == "refine":
        n, it = float(case["n"]), _UPDATES[case["family"]]
        flops = it * (4.0 + case["order"]) * n ** 3
        if case["precision"] not in ("fp64", "fp32"):
            flops += (3.0 + 1.0 + 2.0 + 3.0) * n ** 3  # residual, d^2, update, residual of the refinement
        return {"bytes": (24.0 if case["warm"] else 16.0) * n * n, "flops": flops}
    if op == "batched":
        sizes = np.array(_sizes(case), dtype=np.float64)
        it = 2.0 if case["warm"] else 4.0
        return {"bytes": (24.0 if case["warm"] else 16.0) * float(np.sum(sizes ** 2)),
                "flops": (it * (4.0 + case["order"]) + 3.0 + 3.0) * float(np.sum(sizes ** 3))}
    if op in ("congruence", "residual"):
        n = float(case["n"])
        return {"bytes": 24.0 * n * n, "flops": 3.0 * n ** 3}
    if op == "propose":
        n = float(case["n"])
        return {"bytes": 8.0 * n * n, "flops": n ** 3}
    b = float(case["batch"])
    return {"bytes": 72.0 * b + 5573 * 4.0 * 8, "flops": 6.0 * 5440 * b}


# ------------------------------------------------------------------ the same in 64 bits
def _inv_sqrt(X):
    lam, V = torch.linalg.eigh(X)
    return (V * lam.rsqrt()) @ V.T


def _factor(S, Z0):
    """The limit of the iteration: Z0 (Z0^T S Z0)^{-1/2}; S^{-1/2} from a multiple of the identity."""
    if Z0 is None:
        return _inv_sqrt(S)
    X = Z0.T @ (S @ Z0)
    return Z0 @ _inv_sqrt(0.5 * (X + X.T))


def _mlp64(P, mu, sd, X):
    w = P.split([1024, 64, 4096, 64, 320, 5])
    h = (X - mu) / sd
    h = torch.nn.functional.gelu(h @ w[0].view(64, 16).T + w[1])
    h = torch.nn.functional.gelu(h @ w[2].view(64, 64).T + w[3])
    return h @ w[4].view(5, 64).T + w[5]


def exact(case, seed):
    s, op = prepare(case, seed), case["op"]
    if op == "refine":
        S = s["S"].cuda()
        return {"Z": _factor(S, s["Z0"].cuda() if s["Z0"] is not None else None), "iters": None, "refine_iters": None}
    if op == "batched":
        Z0 = s["Z0"] or [None] * len(s["S"])
        # the residual is that of the Z a run returns, which stops short of the limit
        return {"Z": [_factor(S, z) for S, z in zip(s["S"], Z0)], "resid": None, "iters": None}
    if op == "congruence":
        return {"Hp": s["Z"].T @ (s["H"] @ s["Z"])}
    if op == "residual":
        D = -(s["Z"].T @ (s["S"] @ s["Z"]))
        D.diagonal().add_(1.0)
        return {"D": D, "err": D.norm().reshape(1)}
    if op == "propose":
        S = s["S"]
        n = S.shape[0]
        d, rows = S.diagonal(), S.abs().sum(dim=1)
        off = rows - d.abs()
        g, t1 = (d + off).max(), 1.0 - d.mean() / (d + off).max()
        E = S / -g
        E.diagonal().add_(1.0 - t1)
        E2 = E @ E
        m2, m3, m4 = (E * E).sum() / n, (E2 * E).sum() / n, (E2 * E2).sum() / n
        t2, t3 = m2 + t1 ** 2, m3 + 3 * t1 * m2 + t1 ** 3
        t4 = m4 + 4 * t1 * m3 + 6 * t1 ** 2 * m2 + t1 ** 4
        f = torch.stack([torch.log(torch.full_like(g, n)), g.log(), (d - off).min() / g, d.mean() / g, d.min() / g,
                         rows.mean() / g, rows.min() / g, t1, t2, t3, t4, t2.sqrt(), m2, m3, m4, 0.5 * (t2 * n).log()])
        y = _mlp64(s["P"].double(), s["mu"].double(), s["sd"].double(), f[None])[0]
        s0 = g.rsqrt()
        scale = s0 * y[0].exp()
        return {"scale": (scale if s0 / 4 <= scale <= 4 * s0 else s0).reshape(1), "order": None}
    P = s["P"].double().requires_grad_()
    y = _mlp64(P, s["mu"].double(), s["sd"].double(), s["X"].double())
    loss = ((y[:, 0] - s["ts"].double()) ** 2).mean() + torch.nn.functional.cross_entropy(y[:, 1:], s["to"].long())
    loss.backward()
    grad, P = P.grad, P.detach()
    b1, b2, k = 0.9, 0.999, s["step"]
    M = b1 * s["M"].double() + (1 - b1) * grad
    V = b2 * s["V"].double() + (1 - b2) * grad * grad
    P = P - 1e-3 * (M / (1 - b1 ** k)) / ((V / (1 - b2 ** k)).sqrt() + 1e-8)
    return {"grad": grad, "loss": loss.detach().reshape(1), "P": P, "M": M, "V": V}
