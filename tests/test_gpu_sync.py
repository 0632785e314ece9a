"""Results that depend on an order inside a kernel or between overlapped kernels."""
import numpy as np
import pytest

from paper_1811_11722_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def Q():
    from paper_1811_11722_gb300 import build, qmc
    build.build_library()
    return qmc


@pytest.mark.parametrize("count", [9, 11, 16])
@pytest.mark.parametrize("transform,alpha", [("baker", 0), ("korobov", 3)])
def test_multi_sum_slots(Q, count, transform, alpha):
    """The sum group with an odd shift count (the last launch of a chunk keeps one of its two rows) and a
    short, an odd and a full last chunk: per shift, the integrands' values added.  The two differ in
    the order of at most count + 600 additions of positive numbers: 700 * 2^-53 = 8e-14."""
    probs = I.config3_shared(count=count, d=4, n=50021, m=5, transform=transform, alpha=alpha)
    g = I.random_generating_vector(I.SplitMix64(63), 4, probs[0].n)
    fs = [Q.integrand_from_problem(p, "fp32") for p in probs]
    res, ps = Q.qmc_integrate_multi(4, probs[0].n, 5, g, probs[0].shifts, Q.transform(transform, alpha), fs,
                                    want_per_shift=True)
    assert np.allclose(ps[count, :, 0], ps[:count, :, 0].sum(axis=0), rtol=8e-14, atol=0)
    assert abs(res[count].mean[0] - ps[count, :, 0].mean()) <= 8e-14 * abs(res[count].mean[0])


@pytest.mark.parametrize("d,n_pilot", [(8, 16381), (3, 33013)])
def test_fit_is_reproducible(Q, d, n_pilot):
    """One fit many times: every addition has its place, so parameters and losses keep their bits.  Two sizes: one batch
    of tiles per block of the fit kernel, and several."""
    rng = I.SplitMix64(71 + d)
    U, F = I.random_poly(rng, d, d, 0), I.random_poly(rng, d, 0, min(24, d * (d + 1) // 2))
    f = Q.Integrand(Q.QMC_F_SECTOR, d, Q.QMC_FP32EVAL, (U.coef, U.expo), (F.coef, F.expo))
    g = I.random_generating_vector(rng, d, n_pilot)
    shift = np.array([rng.uniform() for _ in range(d)])
    cfg = Q.qmc_cv_config(16, 32, 1, 60, 1e-2, 0, 5)
    first = None
    for _ in range(30):
        a, losses = Q.qmc_cv_train(d, n_pilot, g, shift, Q.transform("none"), f, cfg)
        got = np.concatenate([np.asarray(a, dtype=np.float64).ravel(), np.asarray(losses, dtype=np.float64).ravel()])
        assert np.all(np.isfinite(got))
        first = got if first is None else first
        assert np.array_equal(got, first)


@pytest.mark.parametrize("m", [8, 1024])
def test_host_results_and_per_shift_values(Q, m):
    """Results and per-shift values wanted on the host together, below and above the size up to which one copy brings
    both: six orders of an epsilon expansion, and the passes of a walk over eight problems."""
    d, n = 3, 1 << 9
    rng = I.SplitMix64(8 + m)
    shifts = I.make_shifts(rng, m, d)
    g = np.array([1, 182667, 469891], dtype=np.uint64)
    U, F = I.random_poly(rng, d, d, 0), I.random_poly(rng, d, 0, 6)
    f = Q.Integrand(Q.QMC_F_SECTOR, d, Q.QMC_FP64, (U.coef, U.expo), (F.coef, F.expo))
    t = Q.transform("korobov", 3)
    res, ps = Q.qmc_integrate_eps(d, n, m, g % n, shifts, t, f, Q.eps_spec(6), want_per_shift=True)
    ps = np.asarray(ps).reshape(6, m, 2)
    for o in range(6):
        assert res[o].status == 0 and np.isclose(res[o].mean[0], ps[o, :, 0].mean(), rtol=1e-13, atol=0)
    levels = 2
    walk, lv, passes, _ = Q.qmc_integrate_batch_extensible([(d, n, m, g % n, shifts, t, f)] * 8, levels, g, 1e-18,
                                                           Q.WALK_EACH)
    assert passes == levels + 1
    last = Q.qmc_integrate(d, n << levels, m, g % (n << levels), shifts, t, f)[0]
    for r in walk:
        assert np.isclose(r.mean[0], last.mean[0], rtol=1e-14, atol=0)
