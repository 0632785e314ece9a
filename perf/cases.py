"""Performance cases of the shifted rank-1 lattice rule, through its public entry points.

A case is a dict of plain values.  ``listed()`` gives the fixed ones, ``draw(rng)``
another of the same ranges.  ``prepare(case, seed)`` makes what a user's program
has in hand before the call (polynomials, generating vector, shift tables, plans,
device buffers), ``run(state)`` is one pass through the library, ``work(case)``
the operations it cannot do without and ``exact(case, seed)`` the same results
from plain FP64 tensor arithmetic, without the library.

Shapes follow the repository's synthetic workloads (``inputs.config1`` ..
``config5`` and the shared-lattice variant): dimensions 2-8, sector integrands
U^-2 F^-1 with linear U and quadratic F, Korobov weight 3 and baker transforms.
Every seed draws new coefficients, monomials, shifts and generating vectors.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1811_11722_gb300 import inputs as I
from paper_1811_11722_gb300 import qmc

CHUNK = 1 << 22  # lattice points per tensor in exact()


# ------------------------------------------------------------------- cases --

def listed():
    return [
        # the plain rule in the paper's arithmetic at its smallest use: one call on a small
        # lattice, results wanted on the host at once (a first look, a check, a control loop)
        dict(name="one_shot_fp64_separable_d3", kind="one_shot", d=3, n=10007, m=10, alpha=3),
        # a sector in double precision, the arithmetic the paper's figures are in, under both transforms
        dict(name="sector_fp64_baker_d6", kind="sector", precision="fp64", transform="baker", d=6, n=1000003, m=32,
             terms_u=6, terms_f=12),
        dict(name="sector_fp64_korobov_d8", kind="sector", precision="fp64", transform="korobov", d=8, n=4194301,
             m=16, terms_u=8, terms_f=24),
        # the throughput workload: FP32 evaluation of one sector on a large lattice
        dict(name="sector_fp32_baker_d6", kind="sector", precision="fp32", transform="baker", d=6, n=16777213, m=32,
             terms_u=6, terms_f=12),
        # the same under the transform that converges fastest, at the largest d with a fast kernel
        dict(name="sector_fp32_korobov_d8", kind="sector", precision="fp32", transform="korobov", d=8, n=16777213,
             m=16, terms_u=8, terms_f=24),
        # finite part and two higher orders of an epsilon expansion in one sweep
        dict(name="eps_fp32_korobov_d6", kind="eps", transform="korobov", d=6, n=4194301, m=16, orders=3, terms_u=6,
             terms_f=12),
        # all sectors of one dimension on one lattice, with their sum
        dict(name="shared_fp32_korobov_d6", kind="multi", transform="korobov", d=6, n=4194301, m=16, count=16),
        # the sectors of one integral, uneven in dimension and size, planned once and replayed
        dict(name="batch_fp32_baker", kind="batch", transform="baker", count=32, m=16, n_lo=100000, n_hi=3000000),
        # the sectors of one integral on embedded lattices, refined by a fixed budget of doublings;
        # in double precision, which targets below about 1e-8 need on base-2 lattices
        dict(name="walk_fp64_korobov", kind="walk", precision="fp64", count=32, m=16, log2_n0=14, levels=3),
        # physical kinematics: the contour-deformed complex integrand in both precisions
        dict(name="deformed_fp64_d5", kind="deformed", precision="fp64", d=5, n=262139, m=20, lam=0.1),
        dict(name="deformed_fp32_d5", kind="deformed", precision="fp32", d=5, n=4194301, m=20, lam=0.1),
        # the learned control variate: fit on a pilot lattice, then the estimator with the fitted surrogate
        dict(name="control_variate_d8", kind="cv", transform="none", d=8, n=2097143, m=16, n_pilot=16381, steps=200),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _terms(rng, d):
    """Term counts of U and F as the batched workload draws them (variables
    without replacement while the count fits)."""
    return rng.randint(min(4, d), min(10, d + 2)), rng.randint(min(6, d * (d + 1) // 2), min(24, d * (d + 1) // 2 + 2))


def draw(rng):
    kind = rng.choice(["one_shot", "sector64", "sector64", "sector32", "sector32", "eps", "multi", "batch", "walk",
                       "deformed64", "deformed32", "cv"])
    d = rng.randint(2, 8)
    tu, tf = _terms(rng, d)
    transform = rng.choice(["baker", "korobov"])
    if kind == "one_shot":
        return dict(kind=kind, d=rng.randint(1, 8), n=_log_int(rng, 1000, 200000), m=rng.randint(8, 20),
                    alpha=rng.choice([1, 2, 3, 3, 3, 4, 6]))
    if kind == "sector64":
        m = rng.randint(8, 32)
        return dict(kind="sector", precision="fp64", transform=transform, d=d, n=_log_int(rng, 20000, 6.4e7 / m), m=m,
                    terms_u=tu, terms_f=tf)
    if kind == "sector32":
        m = rng.randint(16, 32)
        lo = 1e6 if transform == "baker" else 5e6
        return dict(kind="sector", precision="fp32", transform=transform, d=d, n=_log_int(rng, lo, 2.6e8 / m), m=m,
                    terms_u=tu, terms_f=tf)
    if kind == "eps":
        return dict(kind=kind, transform=transform, d=d, n=_log_int(rng, 5e6, 1.2e7), m=16, orders=rng.randint(2, 6),
                    terms_u=tu, terms_f=tf)
    if kind == "multi":
        return dict(kind=kind, transform=transform, d=d, n=_log_int(rng, 4e6, 8e6), m=16, count=rng.randint(5, 16))
    if kind == "batch":
        return dict(kind=kind, transform="baker", count=rng.randint(12, 40), m=16, n_lo=_log_int(rng, 50000, 200000),
                    n_hi=_log_int(rng, 1e6, 4e6))
    if kind == "walk":
        return dict(kind=kind, precision="fp64", count=rng.randint(8, 32), m=16, log2_n0=rng.randint(12, 15),
                    levels=rng.randint(2, 4))
    if kind == "deformed64":
        return dict(kind="deformed", precision="fp64", d=rng.randint(2, 6), n=_log_int(rng, 20000, 500000),
                    m=rng.randint(8, 24), lam=rng.choice([0.05, 0.1, 0.15]))
    if kind == "deformed32":
        return dict(kind="deformed", precision="fp32", d=rng.randint(2, 6), n=_log_int(rng, 6e6, 1.2e7),
                    m=rng.randint(16, 24), lam=rng.choice([0.05, 0.1, 0.15]))
    return dict(kind="cv", transform=rng.choice(["none", "baker", "korobov"]), d=rng.randint(3, 8),
                n=_log_int(rng, 1e6, 4e6), m=16, n_pilot=_log_int(rng, 8000, 33000), steps=rng.randint(100, 300))


# ------------------------------------------------------------------ inputs --

def _transform(name, alpha=3):
    return qmc.transform(name, alpha if name == "korobov" else 0)


def _sector(rng, d, n_lin, n_quad, neg_quad=0):
    return I.random_poly(rng, d, n_lin, 0), I.random_poly(rng, d, 0, n_quad, neg_quad=neg_quad)


def _batch_dims(rng):
    """d, T_U, T_F of one sector as the batched workload draws them."""
    return rng.randint(2, 8), rng.randint(4, 10), rng.randint(6, 20)


def _problems(case, seed):
    """The integration problems of a case: dicts of host values."""
    rng = I.SplitMix64(0x5EED0000 + 7919 * seed)
    k, m = case["kind"], case["m"]
    out = []
    if k == "one_shot":
        d = case["d"]
        c = np.array([rng.uniform() for _ in range(d)])
        b = np.array([rng.uniform() for _ in range(d)])
        out.append(dict(d=d, c=c, b=b, transform="korobov", alpha=case["alpha"]))
    elif k in ("sector", "eps", "cv"):
        d = case["d"]
        tu, tf = (d, min(24, d * (d + 1) // 2)) if k == "cv" else (case["terms_u"], case["terms_f"])
        U, F = _sector(rng, d, tu, tf)
        out.append(dict(d=d, U=U, F=F, transform=case["transform"], alpha=3))
    elif k == "deformed":
        d = case["d"]
        U, F = _sector(rng, d, d, min(2 * d, d * (d + 1) // 2), neg_quad=min(3, d - 1))
        out.append(dict(d=d, U=U, F=F, transform="korobov", alpha=3, lam=case["lam"]))
    elif k == "multi":
        d = case["d"]
        for _ in range(case["count"]):
            U, F = _sector(rng, d, rng.randint(4, 10), rng.randint(6, 20))
            out.append(dict(d=d, U=U, F=F, transform=case["transform"], alpha=3))
    else:  # batch, walk
        lo, hi = (math.log(case["n_lo"]), math.log(case["n_hi"])) if k == "batch" else (0.0, 0.0)
        for _ in range(case["count"]):
            d, tu, tf = _batch_dims(rng)
            U, F = _sector(rng, d, tu, tf)
            n = int(math.exp(rng.uniform_in(lo, hi))) if k == "batch" else 1 << case["log2_n0"]
            out.append(dict(d=d, U=U, F=F, transform="baker" if k == "batch" else "korobov", alpha=3, n=n))
    shared = None
    for p in out:
        p.setdefault("n", case.get("n"))
        p["m"] = m
        if k == "multi" and shared is not None:  # one lattice and one shift table for all integrands
            p["shifts"], p["g"] = shared
            continue
        p["shifts"] = I.make_shifts(rng, m, p["d"])
        p["g"] = I.random_generating_vector(rng, p["d"], p["n"])
        shared = (p["shifts"], p["g"])
    if k == "walk":  # one embedded vector: odd components, the first d of them serve a sector
        g = np.array([1] + [2 * rng.randint(1, (1 << 23) - 1) + 1 for _ in range(7)], dtype=np.uint64)
        for p in out:
            p["g"] = g[:p["d"]]
    if k == "cv":
        p = out[0]
        p["g_pilot"] = I.random_generating_vector(rng, p["d"], case["n_pilot"])
        p["shift_pilot"] = np.array([rng.uniform() for _ in range(p["d"])])
        p["fit_seed"] = seed
    return out


def _integrand(p, precision):
    prec = qmc.QMC_FP64 if precision == "fp64" else qmc.QMC_FP32EVAL
    if "c" in p:
        return qmc.Integrand(qmc.QMC_F_SEPARABLE_EXP, p["d"], prec, c=p["c"], b=p["b"])
    U, F = (p["U"].coef, p["U"].expo), (p["F"].coef, p["F"].expo)
    if "lam" in p:
        return qmc.Integrand(qmc.QMC_F_SECTOR_DEFORMED, p["d"], prec, U, F, lam=p["lam"])
    return qmc.Integrand(qmc.QMC_F_SECTOR, p["d"], prec, U, F)


class _Results:
    """Device memory for `count` results, seen as their fields (qmc_result: mean,
    var and err of both parts as doubles, two counts, the status)."""

    def __init__(self, count):
        words = qmc.RESULT_BYTES // 8
        self.raw = torch.zeros(count, words, dtype=torch.int64, device="cuda")
        self.fields = {"estimate": self.raw.view(torch.float64)[:, :6], "counts": self.raw[:, 6:8],
                       "status": self.raw.view(torch.int32)[:, 16]}


def prepare(case, seed):
    probs = _problems(case, seed)
    k, p = case["kind"], probs[0]
    t = _transform(p["transform"], p["alpha"])
    prec = case.get("precision", "fp64" if k == "one_shot" else "fp32")
    fs = [_integrand(q, prec) for q in probs]
    st = {"kind": k, "probs": probs, "fs": fs, "t": t, "stream": torch.cuda.current_stream().cuda_stream}
    if k == "sector" or k == "deformed" or k == "eps":
        eps = qmc.eps_spec(case["orders"]) if k == "eps" else None
        st["plan"] = qmc.Plan(p["d"], p["n"], p["m"], p["g"], p["shifts"], t, fs[0], eps)
        st["out"] = _Results(case.get("orders", 1))
        # double-precision studies keep the per-shift values, fast sweeps take the estimate
        st["per_shift"] = (torch.zeros(p["m"], 2, dtype=torch.float64, device="cuda") if prec == "fp64" else None)
    elif k == "multi":
        st["plan"] = qmc.MultiPlan(p["d"], p["n"], p["m"], p["g"], p["shifts"], t, fs)
        st["out"] = _Results(len(fs) + 1)
        st["per_shift"] = None
    elif k in ("batch", "walk"):
        st["batch"] = [(q["d"], q["n"], q["m"], q["g"], q["shifts"], t, f) for q, f in zip(probs, fs)]
        if k == "batch":
            st["plan"] = qmc.BatchPlan(st["batch"])
            st["out"] = _Results(len(fs))
            st["per_shift"] = None
        else:
            g = max((q["g"] for q in probs), key=len)
            st["levels"], st["g"] = case["levels"], g
            st["walk_problems"] = [(q["d"], q["n"], q["m"], q["g"] % q["n"], q["shifts"], t, f)
                                   for q, f in zip(probs, fs)]
    elif k == "cv":
        st["cfg"] = qmc.qmc_cv_config(16, 32, 1, case["steps"], 1e-2, 0, p["fit_seed"])
        st["n_pilot"] = case["n_pilot"]
    return st


def _fields(res):
    """A host qmc_result as arrays."""
    return {"estimate": np.array(list(res.mean) + list(res.var) + list(res.err)),
            "counts": np.array([res.nonfinite, res.deform_violations], dtype=np.int64),
            "status": np.array([res.status], dtype=np.int32)}


def run(st):
    k, p = st["kind"], st["probs"][0]
    if k == "one_shot":
        res, ps = qmc.qmc_integrate(p["d"], p["n"], p["m"], p["g"], p["shifts"], st["t"], st["fs"][0],
                                    stream=st["stream"], want_per_shift=True)
        return {**_fields(res), "per_shift": ps}
    if k == "walk":
        # the tolerance is out of reach, so every sector takes its whole budget of doublings
        res, lv, passes, _ = qmc.qmc_integrate_batch_extensible(st["walk_problems"], st["levels"], st["g"], 1e-15,
                                                                qmc.WALK_EACH, stream=st["stream"])
        f = [_fields(r) for r in res]
        return {**{key: np.stack([x[key] for x in f]) for key in f[0]}, "doublings": lv, "passes": passes}
    if k == "cv":
        a, losses = qmc.qmc_cv_train(p["d"], st["n_pilot"], p["g_pilot"], p["shift_pilot"], st["t"], st["fs"][0],
                                     st["cfg"], stream=st["stream"])
        res, ps = qmc.qmc_integrate_cv(p["d"], p["n"], p["m"], p["g"], p["shifts"], st["t"], st["fs"][0], st["cfg"],
                                       a, stream=st["stream"])
        return {**_fields(res), "parameters": a, "losses": losses}
    st["plan"].execute(st["out"].raw, st["per_shift"], stream=st["stream"])
    if st["per_shift"] is not None:
        return {**st["out"].fields, "per_shift": st["per_shift"]}
    return dict(st["out"].fields)


# -------------------------------------------------------------------- work --

def _value_flops(p):
    """Operations of one weighted value: coordinates, U, F, the quotient, the sum."""
    d = p["d"]
    coord = 2 * d if p["transform"] != "korobov" else 14 * d
    if "c" in p:
        return 14 * d + 5 * d + 20
    lin, quad = p["U"].nterms - 1, p["F"].nterms - 1
    if "lam" in p:  # contour, Jacobian determinant, complex U and F
        return coord + 6 * d * d + 8 * d ** 3 // 3 + 4 * lin + 10 * quad + 40
    return coord + 2 * lin + 3 * quad + 4


def work(case):
    probs = _problems(case, 1)
    k, m = case["kind"], case["m"]
    flops, bytes_ = 0.0, 0.0
    for q in probs:
        n = q["n"] << case["levels"] if k == "walk" else q["n"]
        v = _value_flops(q)
        if k == "multi":  # the coordinates are shared
            v -= 14 * q["d"] if q["transform"] == "korobov" else 2 * q["d"]
        if k == "eps":
            v += 10 + 4 * (case["orders"] - 1)
        if k == "cv":  # 16 ranks of a 32-term cosine series per dimension; fit: forward and gradient
            v += q["d"] * (16 * 2 * 32 + 2 * 32 + 16)
            flops += case["steps"] * case["n_pilot"] * q["d"] * 3 * 2 * 16 * 32
            bytes_ += case["n_pilot"] * q["d"] * 32 * 2 * 2
        flops += float(n) * m * v
        bytes_ += 8.0 * (m * q["d"] + q["d"]) + 72.0 + 16.0 * m
    if k == "multi":
        flops += float(probs[0]["n"]) * m * (14 if case["transform"] == "korobov" else 2) * case["d"]
    return {"bytes": bytes_, "flops": flops}


# ------------------------------------------------------------------- exact --

def _coords(p, n, g, k, j):
    """Transformed coordinates and the weight of points j under shift k (Eq. 2, 5, 6)."""
    z, w = [], None
    for i in range(p["d"]):
        x = (j * int(g[i]) % n).double() / n + float(p["shifts"][k, i])
        x = torch.where(x >= 1.0, x - 1.0, x)
        if p["transform"] == "baker":
            z.append(1.0 - (2.0 * x - 1.0).abs())
            continue
        if p["transform"] == "none":
            z.append(x)
            continue
        a = p["alpha"]
        s = torch.minimum(x, 1.0 - x)
        c = math.factorial(2 * a + 1) / math.factorial(a) ** 2
        poly = torch.zeros_like(s)
        for q in range(a, -1, -1):
            poly = poly * s + (-1.0) ** q * c * math.comb(a, q) / (a + q + 1)
        lower = s ** (a + 1) * poly
        z.append(torch.where(x > 0.5, 1.0 - lower, lower))
        f = c * (s * (1.0 - s)) ** a
        w = f if w is None else w * f
    return z, w


def _poly(P, z):
    tot = None
    for c, e in zip(P.coef, P.expo):
        term = None
        for i in range(len(e)):
            for _ in range(int(e[i])):
                term = z[i] if term is None else term * z[i]
        term = torch.full_like(z[0], 1.0 if not z[0].is_complex() else 1.0 + 0j) * float(c) if term is None else term * float(c)
        tot = term if tot is None else tot + term
    return tot


def _deriv(P, k):
    """dP/dz_k as a term table."""
    keep = P.expo[:, k] > 0
    expo = P.expo[keep].copy()
    coef = P.coef[keep] * expo[:, k]
    expo[:, k] -= 1
    return I.Poly(coef, expo)


def _det(A):
    """Determinant of a d x d nested list of tensors (diagonally dominant: no pivoting)."""
    d, A, det = len(A), [list(r) for r in A], None
    for c in range(d):
        det = A[c][c] if det is None else det * A[c][c]
        for r in range(c + 1, d):
            f = A[r][c] / A[c][c]
            for q in range(c + 1, d):
                A[r][q] = A[r][q] - f * A[c][q]
    return det


def _values(p, z, w, orders):
    if "c" in p:
        v, e = torch.ones_like(z[0]), torch.zeros_like(z[0])
        for i in range(p["d"]):
            v = v * (1.0 + float(p["c"][i]) * z[i])
            e = e + float(p["b"][i]) * z[i]
        v = [v * torch.exp(e)]
    elif "lam" in p:
        d, lam = p["d"], p["lam"]
        grads = [_deriv(p["F"], k) for k in range(d)]
        gr = [_poly(G, z) if G.nterms else torch.zeros_like(z[0]) for G in grads]
        wz = [torch.complex(z[k], -lam * z[k] * (1.0 - z[k]) * gr[k]) for k in range(d)]
        J = []
        for k in range(d):
            row = []
            for l in range(d):
                H = _deriv(grads[k], l) if grads[k].nterms else grads[k]
                h = float(H.coef.sum()) if H.nterms else 0.0
                im = -lam * h * z[k] * (1.0 - z[k])
                if k == l:
                    im = im - lam * (1.0 - 2.0 * z[k]) * gr[k]
                row.append(torch.complex(torch.full_like(im, 1.0 if k == l else 0.0), im))
            J.append(row)
        U, F = _poly(p["U"], wz), _poly(p["F"], wz)
        v = [_det(J) / (U * U * F)]
    else:
        U, F = _poly(p["U"], z), _poly(p["F"], z)
        v = [1.0 / (U * U * F)]
        L = torch.log(U) - torch.log(F) if orders > 1 else None
        for o in range(1, orders):
            v.append(v[-1] * L / o)
    return v if w is None else [x * w for x in v]


def _per_shift(p, n, g, orders=1):
    """Q^(k) of every order, [orders, m, 2] (re, im)."""
    q = torch.zeros(orders, p["m"], 2, dtype=torch.float64, device="cuda")
    for j0 in range(0, n, CHUNK):
        j = torch.arange(j0, min(n, j0 + CHUNK), dtype=torch.int64, device="cuda")
        for k in range(p["m"]):
            z, w = _coords(p, n, g, k, j)
            for o, v in enumerate(_values(p, z, w, orders)):
                q[o, k, 0] += v.real.sum()
                if v.is_complex():
                    q[o, k, 1] += v.imag.sum()
    return q / n


def _estimate(q):
    """(mean, var, err) of both parts from per-shift values [..., m, 2]: Eq. (2), (3)."""
    m = q.shape[-2]
    mean = q.mean(dim=-2)
    var = ((q - mean.unsqueeze(-2)) ** 2).sum(dim=-2) / (m * (m - 1))
    return torch.cat([mean, var, var.sqrt()], dim=-1)


def exact(case, seed):
    k = case["kind"]
    if k == "cv":
        return None  # the surrogate comes out of a fit of many rounded steps
    probs = _problems(case, seed)
    none = {"counts": None, "status": None}
    if k in ("batch", "walk"):
        est = []
        for p in probs:
            n = p["n"] << case["levels"] if k == "walk" else p["n"]
            est.append(_estimate(_per_shift(p, n, [int(x) % n for x in p["g"]]))[0])
        more = {"doublings": None, "passes": None} if k == "walk" else {}
        return {"estimate": torch.stack(est), **none, **more}
    if k == "multi":
        q = torch.stack([_per_shift(p, p["n"], p["g"])[0] for p in probs])
        return {"estimate": _estimate(torch.cat([q, q.sum(dim=0, keepdim=True)])), **none}
    p = probs[0]
    q = _per_shift(p, p["n"], p["g"], case.get("orders", 1))
    est = _estimate(q)
    if k == "one_shot":
        return {"estimate": est[0], "counts": None, "status": None, "per_shift": q[0]}
    out = {"estimate": est, **none}
    if case.get("precision") == "fp64":
        out["per_shift"] = q[0]
    return out
