"""The workloads that the library is timed on: one call (or one short run) of each of its main
entry points, over the sizes of its named configurations, ragged sizes between them and the
ranges they span. Inputs follow the recipe of thc_inputs (one log-uniform weight per grid
point, Z = L diag(exp(-k/s)) L^T, N(0,1) start factors), drawn on the GPU."""
import math

import numpy as np
import torch

from paper_2502_17683_gb300 import api

DEV = "cuda"


def listed():
    return [
        # one MTTKRP inside a user's own loop, smallest paper-shaped problem: latency and launches
        dict(name="mttkrp small", op="mttkrp", o=5, v=15, Rt=60, R=80, mode=0, precision="fp64"),
        # the same in the middle of the range (the fit of a small molecule), a virtual mode
        dict(name="mttkrp medium", op="mttkrp", o=20, v=100, Rt=480, R=720, mode=1, precision="fp64"),
        # split-precision MTTKRP at the largest configuration
        dict(name="mttkrp bf16x3 large", op="mttkrp", o=50, v=250, Rt=1200, R=1800, mode=2, precision="bf16x3"),
        # the exact FP64 loss of a given CPD, sizes that are no multiple of a tile
        dict(name="loss ragged", op="loss", o=31, v=147, Rt=713, R=1061),
        # a short FP64 ALS run of the smallest configuration (many such fits are run one by one)
        dict(name="als small", op="als", o=5, v=15, Rt=60, R=80, sweeps=10, precision="fp64"),
        # a short FP64 ALS run of the middle configuration
        dict(name="als medium", op="als", o=20, v=100, Rt=480, R=720, sweeps=4, precision="fp64"),
        # one FP64 sweep with ||G||^2 known, ragged, above the middle
        dict(name="sweep ragged", op="sweep", o=37, v=181, Rt=875, R=1303, precision="fp64"),
        # one sweep of the largest configuration in split precision (the headline workload's step)
        dict(name="sweep bf16x3 large", op="sweep", o=50, v=250, Rt=1200, R=1800, precision="bf16x3"),
        # the normal-equation solve alone, for a virtual mode
        dict(name="solve", op="solve", R=1080, n=150),
        # several uneven problems at once (v = 5o, R_thc = 4(o+v), R_cp = 6(o+v), rounded to 16)
        dict(name="batched", op="batched", nprob=12, o_lo=4, o_hi=30, sweeps=2, shape_seed=0, precision="fp64"),
        # the LT-MP2 exchange energies of a finished CPD
        dict(name="exchange", op="exchange", o=20, v=100, Rt=480, R=720, nalpha=12, emulated=False),
        # the THC core fit from a density-fitted tensor, on the FP64-accurate tensor-core products
        dict(name="core fit", op="core_fit", o=20, v=100, Rt=480, naux=480, emulated=True),
    ]


def _size(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["mttkrp", "mttkrp", "loss", "als", "sweep", "sweep", "solve", "batched", "exchange", "core_fit"])
    if op == "solve":
        return dict(op=op, R=_size(rng, 80, 1800), n=_size(rng, 5, 250))
    o = _size(rng, 5, 50)
    v = max(2, int(o * rng.uniform(3.0, 5.0)))
    Rt = max(8, int((o + v) * rng.uniform(3.0, 4.0)))
    R = max(8, int((o + v) * rng.uniform(4.0, 6.0)))
    if op == "mttkrp":
        return dict(op=op, o=o, v=v, Rt=Rt, R=R, mode=rng.randrange(4), precision=rng.choice(["fp64", "fp64", "bf16x3"]))
    if op == "loss":
        return dict(op=op, o=o, v=v, Rt=Rt, R=R)
    if op == "als":
        sweeps = rng.randrange(2, 6) if o <= 30 else rng.randrange(2, 4)
        return dict(op=op, o=o, v=v, Rt=Rt, R=R, sweeps=sweeps, precision="fp64")
    if op == "sweep":
        return dict(op=op, o=o, v=v, Rt=Rt, R=R, precision=rng.choice(["fp64", "bf16x3"]))
    if op == "batched":
        return dict(op=op, nprob=rng.randrange(3, 13), o_lo=4, o_hi=rng.randrange(8, 27), sweeps=2,
                    shape_seed=rng.randrange(1 << 20), precision="fp64")
    o = min(o, 30)
    v = min(v, 150)
    Rt, R = min(Rt, 720), min(R, 1080)
    if op == "exchange":
        return dict(op=op, o=o, v=v, Rt=Rt, R=R, nalpha=rng.randrange(4, 13), emulated=rng.random() < 0.5)
    return dict(op=op, o=o, v=v, Rt=min(Rt, 480), naux=max(min(Rt, 480), int(3.5 * (o + v))), emulated=rng.random() < 0.5)


# ---- inputs ----------------------------------------------------------------------------
def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(seed)


def _randn(g, *shape):
    return torch.randn(*shape, generator=g, device=DEV, dtype=torch.float64)


def _thc(g, o, v, Rt):
    w = 10.0 ** (2.0 * torch.rand(Rt, generator=g, device=DEV, dtype=torch.float64) - 2.0)
    sc = 1.0 / math.sqrt(Rt)
    Xo, Xv, L = _randn(g, o, Rt) * sc * w, _randn(g, v, Rt) * sc * w, _randn(g, Rt, Rt) * sc
    d = torch.exp(-torch.arange(Rt, device=DEV, dtype=torch.float64) / (Rt / 5.0))
    Z = (L * d) @ L.T
    return Xo, Xv, (0.5 * (Z + Z.T)).contiguous()


def _factors(g, o, v, R):
    return [_randn(g, n, R) for n in (o, v, o, v)]


def _unit(A):
    """Factors with unit columns and the product of the norms, as ALS leaves them."""
    lam = torch.ones(A[0].shape[1], device=DEV, dtype=torch.float64)
    out = []
    for a in A:
        n = torch.linalg.vector_norm(a, dim=0)
        out.append((a / n).contiguous())
        lam = lam * n
    return out, lam


def _batched_shapes(c):
    r = np.random.default_rng([c["shape_seed"], 0xB4])
    up = lambda x: (x + 15) // 16 * 16
    return [(int(o), 5 * int(o), up(24 * int(o)), up(36 * int(o)))
            for o in r.integers(c["o_lo"], c["o_hi"] + 1, size=c["nprob"])]


def _inputs(c, seed):
    g = _gen(seed)
    op = c["op"]
    if op == "solve":
        # H as in ALS: the Hadamard product of three Grams of unit-column factors
        R, n = c["R"], c["n"]
        H = torch.ones(R, R, device=DEV, dtype=torch.float64)
        for m in (max(5, n // 5), n, n):
            a = _randn(g, m, R)
            a = a / torch.linalg.vector_norm(a, dim=0)
            H = H * (a.T @ a)
        return dict(H=H.contiguous(), M=_randn(g, n, R))
    if op == "batched":
        probs = []
        for o, v, Rt, R in _batched_shapes(c):
            Xo, Xv, Z = _thc(g, o, v, Rt)
            probs.append(dict(Xo=Xo, Xv=Xv, Z=Z, A0=_factors(g, o, v, R)))
        return dict(probs=probs)
    o, v, Rt = c["o"], c["v"], c["Rt"]
    Xo, Xv, Z = _thc(g, o, v, Rt)
    s = dict(Xo=Xo, Xv=Xv, Z=Z)
    if op == "core_fit":
        C = _randn(g, c["naux"], Rt) / math.sqrt(Rt)
        B = (C @ (Xo[:, None, :] * Xv[None, :, :]).reshape(o * v, Rt).T).reshape(c["naux"], o, v)
        rms = B.square().mean().sqrt()
        s["B"] = (B + 1e-2 * rms * _randn(g, c["naux"], o, v)).contiguous()
        return s
    s["A0"] = _factors(g, o, v, c["R"])
    if op in ("loss", "exchange"):
        s["A0"], s["lam"] = _unit(s["A0"])
        s["lam"] = s["lam"] * 1e-4
    if op == "exchange":
        # Laplace points of synthetic orbital energies (occupied below, virtual above the gap)
        eo = -0.5 - 1.5 * torch.rand(o, generator=g, device=DEV, dtype=torch.float64)
        ev = 0.2 + 2.8 * torch.rand(v, generator=g, device=DEV, dtype=torch.float64)
        t = torch.logspace(-2, 1, c["nalpha"], dtype=torch.float64, device=DEV)
        s["Lam"] = torch.exp(0.5 * t[:, None] * eo[None, :]).contiguous()
        s["Gam"] = torch.exp(-0.5 * t[:, None] * ev[None, :]).contiguous()
    return s


def _norm2(s):
    S = (s["Xo"].T @ s["Xo"]) * (s["Xv"].T @ s["Xv"])
    return (s["Z"] * (S @ s["Z"] @ S)).sum()


def prepare(case, seed):
    s = _inputs(case, seed)
    s["case"] = case
    op = case["op"]
    if op in ("als", "sweep"):
        s["A"] = [torch.empty_like(a) for a in s["A0"]]
        s["lam"] = torch.ones(case["R"], device=DEV, dtype=torch.float64)
    if op == "sweep":
        s["normG2"] = float(_norm2(s))  # a caller that sweeps by itself computes it once
    if op == "batched":
        for p in s["probs"]:
            p["A"] = [torch.empty_like(a) for a in p["A0"]]
            p["lam"] = torch.ones(p["A0"][0].shape[1], device=DEV, dtype=torch.float64)
    return s


def run(s):
    c = s["case"]
    op = c["op"]
    if op == "mttkrp":
        return api.thc_cpd_mttkrp(s["Xo"], s["Xv"], s["Z"], s["A0"], c["mode"], precision=c["precision"])
    if op == "loss":
        return api.thc_cpd_loss(s["Xo"], s["Xv"], s["Z"], s["A0"], s["lam"])
    if op == "solve":
        return api.thc_cpd_ldl_solve(s["H"], s["M"])[0]
    if op == "exchange":
        return api.thc_cpd_exchange(s["Xo"], s["Xv"], s["Z"], s["A0"], s["lam"], s["Lam"], s["Gam"],
                                    emulated=c["emulated"])
    if op == "core_fit":
        return api.thc_cpd_core_fit(s["Xo"], s["Xv"], s["B"], emulated=c["emulated"])[0]
    if op == "batched":
        for p in s["probs"]:  # every pass from the start factors (they are updated in place)
            for a, a0 in zip(p["A"], p["A0"]):
                a.copy_(a0)
        out = api.thc_cpd_als_batched(s["probs"], c["sweeps"], precision=c["precision"])
        return [[[p["A"], p["lam"]] for p in s["probs"]], np.array([[r["loss"], r["fit"]] for r in out])]
    for a, a0 in zip(s["A"], s["A0"]):
        a.copy_(a0)
    if op == "sweep":
        r = api.thc_cpd_als_sweep(s["Xo"], s["Xv"], s["Z"], s["A"], s["lam"], s["normG2"], precision=c["precision"])
    else:
        r = api.thc_cpd_als(s["Xo"], s["Xv"], s["Z"], s["A"], s["lam"], c["sweeps"], precision=c["precision"])
    return [s["A"], s["lam"], r["loss"], r["fit"]]


# ---- what a pass cannot do without -----------------------------------------------------
def _als_work(o, v, Rt, R, sweeps, norm):
    """Least flops and bytes of `sweeps` sweeps: 4 projections, 2 Z products, 4 back-projections,
    4 symmetric Grams, 4 LDL^T (R^3/3) with two triangular solves (2 n R^2 together)."""
    n = 2 * (o + v)
    per = 2 * 2 * n * Rt * R + 2 * 2 * Rt * Rt * R + n * R * R + 4 * R ** 3 / 3 + 2 * n * R * R
    fl = sweeps * per + (2 * 2 * Rt ** 3 + (o + v) * Rt * Rt if norm else 0)
    by = 8 * ((o + v) * Rt + Rt * Rt + 2 * n * R + R)
    return fl, by


def work(case):
    op = case["op"]
    if op == "solve":
        R, n = case["R"], case["n"]
        return {"bytes": 8 * (R * R + 2 * n * R), "flops": R ** 3 / 3 + 2 * n * R * R}
    if op == "batched":
        w = [_als_work(*sh, case["sweeps"], True) for sh in _batched_shapes(case)]
        return {"bytes": sum(x[1] for x in w), "flops": sum(x[0] for x in w)}
    o, v, Rt = case["o"], case["v"], case["Rt"]
    if op == "core_fit":
        na = case["naux"]
        return {"bytes": 8 * (na * o * v + (o + v) * Rt + Rt * Rt),
                "flops": 2 * na * o * v * Rt + 2 * na * o * Rt + (o + v) * Rt * Rt + Rt ** 3 / 3 + 3 * na * Rt * Rt}
    R, n = case["R"], o + v
    base = 8 * (n * Rt + Rt * Rt + 2 * n * R)
    if op == "mttkrp":
        m = (o, v, o, v)[case["mode"]]
        return {"bytes": base, "flops": 2 * (2 * n - m) * Rt * R + 2 * Rt * Rt * R + 2 * m * Rt * R}
    if op == "loss":
        return {"bytes": base + 8 * R, "flops": 4 * n * Rt * R + 2 * Rt * Rt * R + 2 * n * R * R + n * Rt * Rt + 4 * Rt ** 3}
    if op == "exchange":
        na = case["nalpha"]
        return {"bytes": base + 8 * (R + na * n),
                "flops": na * (4 * n * Rt * R + 2 * Rt * Rt * R + 2 * o * R * R + 2 * v * R * R)}
    fl, by = _als_work(o, v, Rt, R, case.get("sweeps", 1), op == "als")
    return {"bytes": by, "flops": fl}


# ---- the same in plain 64-bit torch ----------------------------------------------------
def _project(X, A):
    return [x.T @ a for x, a in zip(X, A)]


def _mttkrp(s, A, mode):
    X = (s["Xo"], s["Xv"], s["Xo"], s["Xv"])
    W = _project(X, A)
    Y = s["Z"] @ (W[2] * W[3]) if mode < 2 else s["Z"].T @ (W[0] * W[1])
    return X[mode] @ (W[mode ^ 1] * Y)


def _loss(s, A, lam, n2):
    W = _project((s["Xo"], s["Xv"], s["Xo"], s["Xv"]), A)
    inner = (lam * (W[0] * W[1]) * (s["Z"] @ (W[2] * W[3]))).sum()
    G = torch.ones(lam.numel(), lam.numel(), device=DEV, dtype=torch.float64)
    for a in A:
        G = G * (a.T @ a)
    loss = n2 - 2.0 * inner + lam @ (G @ lam)
    return float(loss), float(1.0 - loss.clamp(min=0).sqrt() / n2.sqrt())


def _solve(H, M):
    return torch.cholesky_solve(M.T.contiguous(), torch.linalg.cholesky(H)).T.contiguous()


def _als(s, A, sweeps):
    n2 = _norm2(s)
    A = [a.clone() for a in A]
    for _ in range(sweeps):
        for k in range(4):
            H = torch.ones(A[0].shape[1], A[0].shape[1], device=DEV, dtype=torch.float64)
            for m in range(4):
                if m != k:
                    H = H * (A[m].T @ A[m])
            a = _solve(H, _mttkrp(s, A, k))
            lam = torch.linalg.vector_norm(a, dim=0)
            A[k] = a / torch.where(lam > 0, lam, torch.ones_like(lam))
    return [A, lam, *_loss(s, A, lam, n2)]


def exact(case, seed):
    s = _inputs(case, seed)
    op = case["op"]
    if op == "mttkrp":
        return _mttkrp(s, s["A0"], case["mode"])
    if op == "loss":
        return _loss(s, s["A0"], s["lam"], _norm2(s))
    if op == "solve":
        return _solve(s["H"], s["M"])
    if op == "batched":
        ref = [_als(p, p["A0"], case["sweeps"]) for p in s["probs"]]
        return [[r[:2] for r in ref], np.array([r[2:] for r in ref])]
    if op == "core_fit":
        E = torch.einsum("xia,ip,ap->xp", s["B"], s["Xo"], s["Xv"])
        F = _solve((s["Xo"].T @ s["Xo"]) * (s["Xv"].T @ s["Xv"]), E)
        return F.T @ F
    if op == "exchange":
        A, lam = s["A0"], s["lam"]
        e1 = e2 = 0.0
        for L, G in zip(s["Lam"], s["Gam"]):
            Xo, Xv = s["Xo"] * L[:, None], s["Xv"] * G[:, None]
            U = _project((Xo, Xv, Xo, Xv), A)
            e1 -= float((lam * U[0] * U[3] * (s["Z"] @ (U[2] * U[1]))).sum())
            M1, M3, N = A[0].T @ (L[:, None] * A[0]), A[2].T @ (L[:, None] * A[2]), A[1].T @ (G[:, None] * A[3])
            e2 -= float(lam @ ((M1 * N * M3 * N.T) @ lam))
        return e1, e2, 2.0 * e1 - e2
    return _als(s, s["A0"], case.get("sweeps", 1))
