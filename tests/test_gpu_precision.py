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
