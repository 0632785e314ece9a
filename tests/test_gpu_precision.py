"""Accuracy where a faster evaluation can lose it without any other test noticing:
many integrands, single terms next to the cube's faces, coefficients at the ends of
the ranges that a kernel takes."""
import numpy as np
import pytest

from paper_1811_11722_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def Q():
    from paper_1811_11722_gb300 import build, qmc
    build.build_library()
    return qmc


def random_sector(seed, d, n, m, n_lin, n_quad, **kw):
    rng = I.SplitMix64(0x5EED0000 + 7919 * seed)
    U, F = I.random_poly(rng, d, n_lin, 0), I.random_poly(rng, d, 0, n_quad, neg_quad=kw.pop("neg_quad", 0))
    return I.Problem(f"seed{seed}", d, n, m, I.make_shifts(rng, m, d), U=U, F=F, g=I.random_generating_vector(rng, d, n), **kw)


def estimate(Q, p, precision):
    t = Q.transform(p.transform, p.alpha)
    return Q.qmc_integrate(p.d, p.n, p.m, p.g, p.shifts, t, Q.integrand_from_problem(p, precision))[0]


@pytest.mark.parametrize("seed", [3, 6, 8, 10, 12, 15, 19, 22])
def test_fp32_deformed_estimates(Q, seed):
    """FP32 against FP64 on one lattice, several integrands of the workload.  Over 8.4e7
    values rounding noise alone leaves 8e-10 of |Q| (root mean square of 24 integrands, at most
    1.4e-9); a formula whose roundings are biased for some integrands leaves 4e-9."""
    p = random_sector(seed, 5, 4194301, 20, 5, 10, neg_quad=3, transform="korobov", alpha=3, kind="sector_deformed",
                      aU=-2, aF=-1, lam=0.1)
    a, b = (complex(*estimate(Q, p, prec).mean) for prec in ("fp32", "fp64"))
    assert abs(a - b) <= 2e-9 * abs(b)


def exact_points(p):
    """Untransformed points [n, m, d] of the rule in extended precision."""
    j = np.arange(p.n, dtype=np.uint64)[:, None]
    idx = (j * p.g[None, :].astype(np.uint64)) % np.uint64(p.n)
    x = idx.astype(np.longdouble)[:, None, :] / np.longdouble(p.n) + p.shifts.astype(np.longdouble)[None, :, :]
    return np.where(x >= 1, x - 1, x)


def exact_transform(x, transform):
    """z and the weight of one point, in extended precision."""
    if transform == "none":
        return x, np.longdouble(1)
    s = np.minimum(x, 1 - x)
    if transform == "baker":
        return 2 * s, np.longdouble(1)
    low = s ** 4 * (35 + s * (-84 + s * (70 - 20 * s)))
    u = s * (1 - s)
    return np.where(x > 0.5, 1 - low, low), np.prod(140 * u * u * u, axis=-1)


def exact_poly(P, z):
    tot = np.zeros(z.shape[:-1], dtype=np.longdouble)
    for c, e in zip(P.coef, P.expo):
        term = np.full_like(tot, np.longdouble(c))
        for i in np.nonzero(e)[0]:
            term = term * z[..., i] ** int(e[i])
        tot += term
    return tot


@pytest.mark.parametrize("transform", ["none", "baker", "korobov"])
@pytest.mark.parametrize("linear", [0, 2])
@pytest.mark.parametrize("d", [1, 2, 3, 5, 8])
def test_fp64_peaked_sectors(Q, d, transform, linear):
    """FP64 sectors whose constant term is 1/990 of the coefficients' sum R, against extended precision:
    the integrand peaks at the cube's corner, where U and F are a thousandth of their
    range and (Korobov) the weight is small.  What may be left: half a unit of U's and F's constants, 2 R
    2^-64 + R 2^-63 together 2.2e-16, and four roundings of the sum, the scale and the mean, 4.4e-16."""
    rng = I.SplitMix64(500 + 10 * d + linear)
    U, F = I.random_poly(rng, d, d, 0), I.random_poly(rng, d, min(linear, d), d * (d + 1) // 2)
    for P in (U, F):
        P.coef[0] = P.coef[1:].sum() / 989.0
    n, m = 65537, 4
    p = I.Problem("peak", d, n, m, I.make_shifts(rng, m, d), transform, alpha=3 if transform == "korobov" else 0, U=U,
                  F=F, g=I.random_generating_vector(rng, d, n))
    z, w = exact_transform(exact_points(p), transform)
    ref = (w / (exact_poly(U, z) ** 2 * exact_poly(F, z))).mean()
    got = estimate(Q, p, "fp64").mean[0]
    assert abs(got - ref) <= 6.6e-16 * abs(ref), float(got / ref - 1)


@pytest.mark.parametrize("d", [1, 3, 6, 8])
@pytest.mark.parametrize("jit", ["1", "0"])
def test_fp32_single_terms_next_to_faces(Q, monkeypatch, d, jit):
    """Listed FP32 terms with one coordinate 0.1 to 1e-6 from a face (point 0, which has no dither, under shifts that
    lie there; two such coordinates' weights would leave float's range): relative to the same value at the
    coordinate used, at most 3 (2 d + 2) roundings of 2^-24 in the weight's cube and 3 (2 d + 12) in U^-2 F^-1,
    whatever the weight's size."""
    monkeypatch.setenv("QMC_JIT", jit)
    rng = I.SplitMix64(900 + d)
    m, n = 64, 10007
    U, F = I.random_poly(rng, d, d, 0), I.random_poly(rng, d, 0, d * (d + 1) // 2)
    U.coef[0] = F.coef[0] = 2.0
    shifts = np.array([[rng.uniform_in(0.2, 0.8) for _ in range(d)] for _ in range(m)])
    for k in range(m):
        near = 10.0 ** -rng.uniform_in(1, 6)
        shifts[k, k // 2 % d] = 1.0 - near if k % 2 else near
    p = I.Problem("faces", d, n, m, shifts, "korobov", alpha=3, U=U, F=F, g=I.random_generating_vector(rng, d, n))
    f, t = Q.integrand_from_problem(p, "fp32"), Q.transform("korobov", 3)
    j, k = np.zeros(m, dtype=np.uint64), np.arange(m, dtype=np.int32)
    v, _, x = Q.qmc_sample_points(d, n, m, p.g, shifts, t, f, j, k)
    assert np.all(np.abs(x - shifts) <= 2.0 ** -33)  # rounded to 32 bits
    z, w = exact_transform(x.astype(np.longdouble), "korobov")
    uu, ff = exact_poly(U, z), exact_poly(F, z)
    ref = w / (uu * uu * ff)
    tol = (3 * (2 * d + 2) + 3 * (2 * d + 12)) * 2.0 ** -24
    assert np.all(np.abs(v[:, 0] - ref) <= tol * ref), float(np.max(np.abs(v[:, 0] / ref - 1)))
    e = Q.qmc_sample_points_eps(d, n, m, p.g, shifts, t, f, Q.eps_spec(3), j, k)
    assert np.all(np.abs(e[:, 0] - ref) <= tol * ref), float(np.max(np.abs(e[:, 0] / ref - 1)))


def exact_deformed(p):
    """Weighted values of the contour-deformed integrand at every point and shift, in extended precision."""
    y, w = exact_transform(exact_points(p), p.transform)
    d, lam = p.d, np.longdouble(p.lam)
    H = np.zeros((d, d))
    lin = np.zeros(d)
    for c, e in zip(p.F.coef, p.F.expo):
        v = [i for i in range(d) for _ in range(int(e[i]))]
        if len(v) == 1:
            lin[v[0]] += c
        elif len(v) == 2:
            H[v[0], v[1]] += c
            H[v[1], v[0]] += c
    grad = [lin[k] + sum(np.longdouble(H[k, l]) * y[..., l] for l in range(d)) for k in range(d)]
    a = [y[..., k] * (1 - y[..., k]) for k in range(d)]
    z = np.stack([y[..., k] - 1j * (lam * a[k] * grad[k]) for k in range(d)], axis=-1)
    J = [[(1 if k == l else 0) - 1j * (lam * (H[k, l] * a[k] + ((1 - 2 * y[..., k]) * grad[k] if k == l else 0)))
          for l in range(d)] for k in range(d)]
    det = np.ones(z.shape[:-1], dtype=z.dtype)
    for c in range(d):  # diagonally dominant: no pivoting
        det = det * J[c][c]
        for r in range(c + 1, d):
            f = J[r][c] / J[c][c]
            for q in range(c + 1, d):
                J[r][q] = J[r][q] - f * J[c][q]

    def poly(P):
        tot = np.zeros(z.shape[:-1], dtype=z.dtype)
        for c, e in zip(P.coef, P.expo):
            term = np.full_like(tot, np.longdouble(c))
            for i in np.nonzero(e)[0]:
                term = term * z[..., i] ** int(e[i])
            tot = tot + term
        return tot
    return w * det / (poly(p.U) ** 2 * poly(p.F))


def deformed_problem(d, ratio, lam, linear, n=20011, m=4):
    rng = I.SplitMix64(1000 * d + ratio + int(100 * lam) + 7 * linear)
    U = I.random_poly(rng, d, d, 0)
    F = I.random_poly(rng, d, d if linear else 0, d * (d + 1) // 2, neg_quad=min(1, d - 1))
    for P in (U, F):
        P.coef[0] = np.abs(P.coef[1:]).sum() / (ratio - 1)
    return I.Problem("def", d, n, m, I.make_shifts(rng, m, d), "korobov", alpha=3, kind="sector_deformed", U=U, F=F,
                     aU=-2, aF=-1, lam=lam, g=I.random_generating_vector(rng, d, n))


@pytest.mark.parametrize("d,ratio,lam,linear", [(1, 950, 0.02, 1), (1, 950, 0.4, 1), (2, 950, 0.1, 1), (2, 950, 0.4, 0),
                                                (7, 4, 0.4, 0), (7, 950, 0.1, 1)])
def test_fp64_deformed_in_double(Q, d, ratio, lam, linear):
    """FP64 deformed integrands outside of the fixed-point form's range (coordinates in fixed point, the rest in double)
    against extended precision: six roundings of 2^-53 for the sum, the scale, the mean and the constants."""
    p = deformed_problem(d, ratio, lam, linear)
    ref = exact_deformed(p).mean()
    got = complex(*estimate(Q, p, "fp64").mean)
    assert abs(got - ref) <= 6.7e-16 * abs(ref), float(abs(got - ref) / abs(ref))


@pytest.mark.parametrize("d,b", [(1, -20.0), (1, -1e3), (1, -1e6), (1, -1e8), (2, -1e3), (3, -100.0)])
def test_fp64_separable_peaks(Q, d, b):
    """FP64 separable exponentials that peak at z = 0, against extended precision: six roundings of 2^-53 for the sum, the
    scale, the mean and the factors (those of the exponents, which are small where the values are large, average out)."""
    rng = I.SplitMix64(5000 + d)
    n, m = 20011, 4
    p = I.Problem("peak", d, n, m, I.make_shifts(rng, m, d), "korobov", alpha=3, kind="separable_exp",
                  b=b * np.array([rng.uniform_in(0.5, 1) for _ in range(d)]), c=np.zeros(d),
                  g=I.random_generating_vector(rng, d, n))
    z, w = exact_transform(exact_points(p), "korobov")
    ref = (w * np.exp((p.b.astype(np.longdouble) * z).sum(axis=-1))).mean()
    got = estimate(Q, p, "fp64").mean[0]
    assert abs(got - ref) <= 6.7e-16 * abs(ref), float(got / ref - 1)


@pytest.mark.parametrize("kind", ["const", "separable_exp", "trig"])
@pytest.mark.parametrize("near", [1e-2, 1e-3, 1e-4])
def test_fp64_separable_small_weights(Q, kind, near):
    """A rule of three points each of which has five of its fifteen coordinates next to a face: the weights, down to
    1e-49 of the largest, keep their relative precision: three roundings for each of 15 factors and fifteen for
    the sum, 6.7e-15 (a factor's own error, a unit of 2^-64 in 4e-4, is below them)."""
    d, n, m = 15, 3, 2
    shifts = np.array([[(i % 3) / 3 + near * (1 + 0.1 * i) for i in range(d)], [(i % 3) / 3 + near * (2 - 0.05 * i) for i in range(d)]])
    p = I.Problem("small", d, n, m, shifts, "korobov", alpha=3, kind=kind, c=np.zeros(d), b=np.zeros(d),
                  h=np.zeros(d, dtype=np.int32), g=np.ones(d, dtype=np.uint64))
    _, w = exact_transform(exact_points(p), "korobov")
    _, ps = Q.qmc_integrate(d, n, m, p.g, shifts, Q.transform("korobov", 3), Q.integrand_from_problem(p, "fp64"),
                            want_per_shift=True)
    ref = w.mean(axis=0)
    assert np.all(np.abs(ps[:, 0] - ref) <= 6.7e-15 * ref), (ps[:, 0], ref)


@pytest.mark.parametrize("d,ratio,lam,linear", [(1, 64, 0.1, 0), (1, 400, 0.02, 0), (1, 400, 0.4, 1), (2, 400, 0.4, 1),
                                                (3, 4, 0.1, 0), (3, 400, 0.4, 0), (4, 64, 0.4, 1), (5, 4, 0.4, 0),
                                                (5, 16, 0.1, 1), (6, 4, 0.15, 1), (6, 64, 0.02, 0)])
def test_fp64_deformed_estimates(Q, d, ratio, lam, linear):
    """FP64 deformed estimates against extended precision, small and large deformations, constants from 1/4 to 1/400 of
    the coefficients' sum: six roundings of 2^-53 for the sum, the scale, the mean and the fixed-point scales."""
    p = deformed_problem(d, ratio, lam, linear)
    ref = exact_deformed(p).mean()
    got = complex(*estimate(Q, p, "fp64").mean)
    assert abs(got - ref) <= 6.7e-16 * abs(ref), float(abs(got - ref) / abs(ref))


@pytest.mark.parametrize("d", [2, 5, 8])
def test_fp32_centred_form_at_its_line(Q, monkeypatch, d):
    """The FP32 Korobov coordinate centred on x = 1/2 serves constants down to 2^-d (from d = 5 on 2^-(d + 1)) of the
    coefficients' sum: there its estimates have to be as near to FP64 as those of the plain form, which takes
    the same integrands with a constant 0.2 % smaller.  Root mean square of eight integrands over 1.3e8 values
    each (the forms' noise differs by 0.6, the sample's by 0.25)."""
    monkeypatch.setenv("QMC_JIT", "0")
    n, m = 4194301, 32
    line = 2.0 ** (d if d <= 4 else d + 1)
    rms = []
    for ratio in (0.999 * line, 1.001 * line):
        rel = []
        for s in range(8):
            rng = I.SplitMix64(40 * d + s)
            U, F = I.random_poly(rng, d, d, 0), I.random_poly(rng, d, 0, d * (d + 1) // 2)
            for P in (U, F):
                P.coef[0] = np.float32(P.coef[1:].sum() / (ratio - 1))
            p = I.Problem("line", d, n, m, I.make_shifts(rng, m, d), "korobov", alpha=3, U=U, F=F,
                          g=I.random_generating_vector(rng, d, n))
            a, b = (estimate(Q, p, prec).mean[0] for prec in ("fp32", "fp64"))
            rel.append((a - b) / b)
        rms.append(float(np.sqrt(np.mean(np.square(rel)))))
    assert rms[0] <= rms[1], rms


def described(Q, p, precision="fp64"):
    return Q.Plan(p.d, p.n, p.m, p.g, p.shifts, Q.transform(p.transform, p.alpha),
                  Q.integrand_from_problem(p, precision)).describe()


@pytest.mark.parametrize("case,fixed", [
    (dict(d=3), 1), (dict(d=6), 1), (dict(d=7), 0), (dict(d=3, aU=-1), 0), (dict(d=3, quad_u=2), 0), (dict(d=3, alpha=2), 0),
    (dict(d=3, f0=1 / 240), 1), (dict(d=3, f0=1 / 260), 0), (dict(d=3, u0=1 / 240), 1), (dict(d=3, u0=1 / 260), 0),
    (dict(d=2, gsum=1.05 / 32), 1), (dict(d=2, gsum=0.95 / 32), 0), (dict(d=1, gsum=3.9), 1), (dict(d=1, gsum=4.1), 0)])
def test_deformed_dispatch(Q, case, fixed):
    """Which FP64 deformed plans are evaluated in fixed point: either side of every limit that one integrand can be put at
    (f0, u0: the constant over the sum it is held against; gsum: the largest sum of |lambda dF|)."""
    d = case["d"]
    rng = I.SplitMix64(31 + d)
    U = I.random_poly(rng, d, d, case.get("quad_u", 0))
    F = I.random_poly(rng, d, d, d * (d + 1) // 2)
    coefs = 2.0 * F.coef[1:].sum()  # sum of |dF(0)| twice and of the Hessian's entries
    F.coef[0] = case.get("f0", 1.0) * coefs
    U.coef[0] = case.get("u0", 1.0) * U.coef[1:].sum()
    grads = sum(2 * c if e.sum() == 2 else c for c, e in zip(F.coef[1:], F.expo[1:]))
    p = I.Problem("def", d, 1021, 4, I.make_shifts(rng, 4, d), "korobov", alpha=case.get("alpha", 3),
                  kind="sector_deformed", U=U, F=F, aU=case.get("aU", -2), aF=-1,
                  lam=case["gsum"] / grads if "gsum" in case else 0.05, g=I.random_generating_vector(rng, d, 1021))
    assert described(Q, p)["fixed"] == str(fixed)


def test_plan_description_of_fixed_point_plans(Q):
    """Points per thread and tile are told for every kind of plan, as before the fixed-point kernels."""
    for d, kind in ((4, {}), (3, dict(kind="sector_deformed", aU=-2, aF=-1, lam=0.05))):
        p = random_sector(3, d, 1000003, 8, d, d, transform="korobov", alpha=3, **kind)
        desc = described(Q, p)
        assert desc["fixed"] == "1" and int(desc["L"]) >= 1


def test_fp32_epsilon_estimates(Q):
    """Three epsilon orders of one integrand over 6.7e7 FP32 values, as recorded with the plain Korobov coordinate, to the
    sums' rounding.  The coordinate centred on x = 1/2 moves this integrand's by 1.1e-9."""
    p = random_sector(10, 6, 4194301, 16, 6, 12, transform="korobov", alpha=3)
    res, _ = Q.qmc_integrate_eps(p.d, p.n, p.m, p.g, p.shifts, Q.transform("korobov", 3),
                                 Q.integrand_from_problem(p, "fp32"), Q.eps_spec(3))
    recorded = [0.018633754043793173, -0.010577168001121313, 0.003257045716876482]
    assert np.allclose([r.mean[0] for r in res], recorded, rtol=1e-11, atol=0)
