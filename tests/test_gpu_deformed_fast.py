"""The deformed FAST kernels (det J from principal minors, F from its gradient)
against the oracle's pivoted LU: every dimension they take and the first above,
both coordinate forms, odd and many shifts, ragged and tiny lattices, U of degree 2
and other powers.

Tolerances are those of the full-size tests: FP64 1e-12, FP32 2e-6 of |Q^(k)| (the
FP32 sums here are short, so single values' rounding, up to 3e-5 on a vanishing
one, averages over at least 2 10^4 points or is allowed for by 2e-5)."""
import numpy as np
import pytest

from paper_1811_11722_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def Q():
    from paper_1811_11722_gb300 import build, qmc
    build.build_library()
    return qmc


def run(Q, oracle_lib, nthreads, d, n, m, precision, tol, c0=None, quad_u=0, powers=(-2, -1), lam=0.1):
    rng = I.SplitMix64(31 * d + n + m)
    U = I.random_poly(rng, d, d, quad_u)
    F = I.random_poly(rng, d, 1 if d > 1 else 0, min(2 * d, d * (d + 1) // 2), neg_quad=1)
    if c0 is not None:
        for P in (U, F):
            P.coef[0] = float(np.float32(c0))
    p = I.Problem("def", d, n, m, I.make_shifts(rng, m, d), "korobov", alpha=3, kind="sector_deformed", U=U, F=F,
                  aU=powers[0], aF=powers[1], lam=lam, g=I.random_generating_vector(rng, d, n))
    f = Q.integrand_from_problem(p, precision)
    res, ps = Q.qmc_integrate(d, n, m, p.g, p.shifts, Q.transform("korobov", 3), f, want_per_shift=True)
    ref = oracle_lib.integrate(p, p.g, nthreads=nthreads)
    a, b = ps[:, 0] + 1j * ps[:, 1], ref["q"][:, 0] + 1j * ref["q"][:, 1]
    assert np.all(np.abs(a - b) <= tol * np.abs(b)), np.abs(a / b - 1).max()
    assert res.deform_violations == 0 and res.nonfinite == 0


@pytest.mark.parametrize("precision,tol", [("fp64", 1e-12), ("fp32", 2e-6)])
@pytest.mark.parametrize("d", range(1, 9))
def test_dimensions(Q, oracle_lib, nthreads, d, precision, tol):
    run(Q, oracle_lib, nthreads, d, 20011 + d, 5, precision, tol, lam=0.05)


@pytest.mark.parametrize("precision,tol", [("fp64", 1e-12), ("fp32", 2e-5)])
@pytest.mark.parametrize("n,m", [(2, 2), (257, 33), (1021, 3), (50021, 40)])
def test_sizes(Q, oracle_lib, nthreads, n, m, precision, tol):
    run(Q, oracle_lib, nthreads, 3, n, m, precision, tol)


@pytest.mark.parametrize("c0", [4.0, 0.12])
def test_both_coordinate_forms(Q, oracle_lib, nthreads, c0):
    run(Q, oracle_lib, nthreads, 4, 30011, 6, "fp32", 2e-6, c0=c0)


@pytest.mark.parametrize("precision,tol", [("fp64", 1e-12), ("fp32", 2e-6)])
@pytest.mark.parametrize("quad_u,powers", [(2, (-2, -1)), (0, (-1, -2)), (2, (1, -1))])
def test_quadratic_u_and_powers(Q, oracle_lib, nthreads, precision, tol, quad_u, powers):
    run(Q, oracle_lib, nthreads, 4, 20021, 9, precision, tol, quad_u=quad_u, powers=powers)


@pytest.mark.parametrize("d,c0,lam,linear", [(1, 2.0, 0.3, True), (3, 2.0, 0.3, False), (5, 0.5, 0.1, False),
                                             (6, 1.0, 0.02, True), (6, 0.01, 0.05, True), (4, 1.0, 1e-4, True),
                                             (5, 2.0, 0.45, True), (6, 2.0, 1.5, False)])
def test_fixed_point_ranges(Q, oracle_lib, nthreads, d, c0, lam, linear):
    """The fixed-point FP64 form at the ends of its scales, and integrands just
    outside of it (a small constant, a small or a large lambda)."""
    rng = I.SplitMix64(977 * d + int(1000 * lam))
    U = I.random_poly(rng, d, d, 0)
    F = I.random_poly(rng, d, d if linear else 0, d * (d + 1) // 2, neg_quad=0)
    U.coef[0], F.coef[0] = 1.0, float(np.float32(c0))
    n, m = 30011, 7
    p = I.Problem("def", d, n, m, I.make_shifts(rng, m, d), "korobov", alpha=3, kind="sector_deformed", U=U, F=F,
                  aU=-2, aF=-1, lam=lam, g=I.random_generating_vector(rng, d, n))
    f = Q.integrand_from_problem(p, "fp64")
    _, ps = Q.qmc_integrate(d, n, m, p.g, p.shifts, Q.transform("korobov", 3), f, want_per_shift=True)
    ref = oracle_lib.integrate(p, p.g, nthreads=nthreads)
    a, b = ps[:, 0] + 1j * ps[:, 1], ref["q"][:, 0] + 1j * ref["q"][:, 1]
    assert np.all(np.abs(a - b) <= 1e-12 * np.abs(b)), np.abs(a / b - 1).max()
