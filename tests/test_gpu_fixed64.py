"""The fixed-point FP64 kernels (sectors, separable integrands) against the oracle where they can go wrong:
every dimension and transform, ragged tiles and odd shift counts, coefficients
that use all 53 bits, constant terms at both sides of the range the kernel
takes, single terms with tiny weights.

Tolerance: the fixed-point value is good to 2^-56, so the difference is the
oracle's own rounding, at most (d + terms) roundings of 2^-53 in U, F and the
weight, three powers of each: 3 * 60 * 2^-53 = 2e-14 relative on positive sums."""
import dataclasses

import numpy as np
import pytest

from paper_1811_11722_gb300 import inputs as I

pytestmark = pytest.mark.gpu
TOL = 2e-14


@pytest.fixture(scope="module")
def Q():
    from paper_1811_11722_gb300 import build, qmc
    build.build_library()
    return qmc


def problem(d, n, m, transform, seed, c0=None):
    rng = I.SplitMix64(seed)
    U, F = I.random_poly(rng, d, d, 0), I.random_poly(rng, d, 0, d * (d + 1) // 2)
    for P in (U, F):  # full-mantissa coefficients
        P.coef[:] = [rng.uniform_in(0.1, 2.0) for _ in range(P.nterms)]
        if c0 is not None:
            P.coef[0] = P.coef[1:].sum() * c0
    return I.Problem(f"fx_d{d}", d, n, m, I.make_shifts(rng, m, d), transform, alpha=3 if transform == "korobov" else 0,
                     U=U, F=F, g=I.random_generating_vector(rng, d, n))


def check(Q, oracle_lib, p, fixed, nthreads=1):
    f = Q.integrand_from_problem(p, "fp64")
    plan = Q.Plan(p.d, p.n, p.m, p.g, p.shifts, Q.transform(p.transform, p.alpha), f)
    assert (plan.describe()["shifts_per_launch"] == "32") == fixed
    ps = np.zeros((p.m, 2))
    res = plan.execute(per_shift=ps)
    ref = oracle_lib.integrate(p, p.g, nthreads=nthreads)
    assert res.status == 0 and res.nonfinite == 0
    assert np.all(np.abs(ps[:, 0] - ref["q"][:, 0]) <= TOL * np.abs(ref["q"][:, 0])), (ps[:, 0], ref["q"][:, 0])
    assert abs(res.mean[0] - ref["mean"][0]) <= TOL * abs(ref["mean"][0])


@pytest.mark.parametrize("d", range(1, 9))
@pytest.mark.parametrize("transform", ["none", "baker", "korobov"])
def test_dimensions(Q, oracle_lib, nthreads, d, transform):
    check(Q, oracle_lib, problem(d, 20011 + d, 5, transform, 100 * d), True, nthreads)


@pytest.mark.parametrize("n,m", [(2, 2), (255, 3), (256, 2), (257, 32), (513, 33), (300007, 65)])
def test_sizes(Q, oracle_lib, nthreads, n, m):
    check(Q, oracle_lib, problem(4, n, m, "korobov", n + m), True, nthreads)


@pytest.mark.parametrize("c0,fixed", [(0.5, True), (1 / 990.0, True), (1 / 1005.0, False)])
@pytest.mark.parametrize("transform", ["none", "baker", "korobov"])
def test_constant_term_range(Q, oracle_lib, nthreads, c0, fixed, transform):
    """c0 is the constant over the other coefficients' sum: the kernel takes sum / constant <= 1000."""
    check(Q, oracle_lib, problem(5, 40009, 4, transform, 77, c0), fixed, nthreads)


def test_terms(Q, oracle_lib):
    """Single terms, the smallest weights of 4096 random points among them."""
    p = problem(6, 1000003, 8, "korobov", 5)
    rng = np.random.default_rng(1)
    j, k = rng.integers(0, p.n, 4096).astype(np.uint64), rng.integers(0, p.m, 4096).astype(np.int32)
    v, idx, x = Q.qmc_sample_points(p.d, p.n, p.m, p.g, p.shifts, Q.transform("korobov", 3),
                                    Q.integrand_from_problem(p, "fp64"), j, k)
    order = np.argsort(np.abs(v[:, 0]))
    for s in list(order[:100]) + list(order[-20:]):
        ref, oi, ox, _, _ = oracle_lib.point(p, p.g, int(k[s]), int(j[s]))
        assert np.array_equal(idx[s], oi)
        # the oracle's coordinate carries 2^-52; the weight's sensitivity to it is 3 dx / s per factor
        rel = TOL + float(np.sum(6.0 * 2.0 ** -52 / np.minimum(ox, 1.0 - ox)))
        assert abs(v[s, 0] - ref[0]) <= rel * abs(ref[0])


def test_moves_with_the_walk(Q):
    """Capped grids, moved lattices and moved shifts: the embedded walk in double precision ends on the rule of its size."""
    m, n0, levels = 6, 1 << 9, 3
    g = np.array([1, 182667, 469891, 498753], dtype=np.uint64)
    ps = [problem(d, n0, m, "korobov", 40 + d) for d in (2, 3, 4)]
    probs = [(p.d, n0, m, g[:p.d] % n0, p.shifts, Q.transform("korobov", 3), Q.integrand_from_problem(p, "fp64"))
             for p in ps]
    res, lv, passes, _ = Q.qmc_integrate_batch_extensible(probs, levels, g, 1e-18, Q.WALK_EACH)
    assert list(lv) == [levels] * 3 and passes == levels + 1
    for p, r in zip(ps, res):
        n = n0 << levels
        q = dataclasses.replace(p, n=n, g=g[:p.d] % n)
        d, _ = Q.qmc_integrate(q.d, n, m, q.g, q.shifts, Q.transform("korobov", 3), Q.integrand_from_problem(q, "fp64"))
        assert abs(r.mean[0] - d.mean[0]) <= 1e-15 * abs(d.mean[0])


@pytest.mark.parametrize("kind", ["const", "separable_exp", "trig"])
@pytest.mark.parametrize("transform,alpha", [("none", 0), ("baker", 0), ("korobov", 3), ("korobov", 5)])
@pytest.mark.parametrize("d,n,m", [(1, 2, 2), (3, 257, 33), (7, 10007, 5), (16, 65537, 40)])
def test_separable(Q, oracle_lib, nthreads, kind, transform, alpha, d, n, m):
    """Sums of both signs (trig) are held to the largest term: 1 without a
    weight, Eq. (5)'s largest weight (35/16 at alpha = 3, 2.71 at 5) to the power d with one,
    over sqrt(n) terms' worth of rounding and never below one."""
    rng = I.SplitMix64(n + 7 * d)
    p = I.Problem("sep", d, n, m, I.make_shifts(rng, m, d), transform, alpha=alpha, kind=kind,
                  c=np.array([rng.uniform_in(-0.5, 1.0) for _ in range(d)]),
                  b=np.array([rng.uniform_in(-0.5, 0.5) for _ in range(d)]),
                  h=np.array([rng.randint(-3, 3) for _ in range(d)], dtype=np.int32),
                  g=I.random_generating_vector(rng, d, n))
    f = Q.integrand_from_problem(p, "fp64")
    res, ps = Q.qmc_integrate(d, n, m, p.g, p.shifts, Q.transform(transform, alpha), f, want_per_shift=True)
    ref = oracle_lib.integrate(p, p.g, nthreads=nthreads)
    assert res.status == 0 and res.nonfinite == 0
    top = {0: 1.0, 3: 35.0 / 16.0, 5: 2.71}[alpha] ** d / np.sqrt(n) if kind == "trig" else 0.0
    tol = 20 * (d + 2) * 2.0 ** -53
    assert np.all(np.abs(ps[:, 0] - ref["q"][:, 0]) <= tol * np.maximum(np.abs(ref["q"][:, 0]), max(top, 1.0) if kind == "trig" else 0.0))
