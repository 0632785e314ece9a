// Plans of FP64 integrands on the fixed-point kernels (sectors: fixed64.cuh,
// deformed: deformed_fx.cuh): which integrands they take, the coefficients in
// fixed point, the launches.
#include <algorithm>
#include <cmath>
#include <cstring>

#include "fixed64.cuh"
#include "plan.h"

namespace qmc {

namespace {

// c 2^k as (high word, low word / 16), rounded to the nearest multiple of 16
void fx_split(double c, int k, uint32_t* h, uint32_t* l) {
  const uint64_t q = (uint64_t)std::llrint(std::ldexp(c, k - 4));
  *h = (uint32_t)(q >> 28);
  *l = (uint32_t)(q & 0x0FFFFFFFu);
}

// c 2^k + more, rounded once
uint64_t fx_fixed(double c, int k, double more) {
  const double q = std::ldexp(c, k), whole = std::floor(q);
  return (uint64_t)whole + (uint64_t)std::llrint((q - whole) + more);
}

// k with sum(c) 2^k in [2^62, 2^64), kept clear of 2^64 by rounding, and the ratio
// of the sum to the constant term; false when that is too large or the scale is
// extreme.
bool fx_scale(const std::vector<double>& c, int* k, double* ratio) {
  double sum = 0.0;
  for (double v : c) sum += v;
  if (!(c[0] > 0.0) || !std::isfinite(sum) || c[0] * kFxRange < sum) return false;
  int x = 0;
  const double f = std::frexp(sum, &x);
  *k = 64 - x - (f > 1.0 - 0x1p-30 ? 1 : 0);
  *ratio = sum / c[0];
  return std::abs(*k) <= 200;
}

void fx_lattice(FxBase& P, uint64_t n, const uint64_t* g) {
  P.n = n;
  P.rc = reciprocal(n);
  for (int i = 0; i < P.d; ++i) {
    P.g[i] = (uint32_t)g[i];
    const uint64_t idx = ((uint64_t)kThreads * g[i]) % n;
    const unsigned __int128 lo = (unsigned __int128)idx * P.rc.rlo;
    const uint64_t top = idx * P.rc.rhi + (uint64_t)(lo >> 64);
    P.step[i][0] = (uint32_t)((uint64_t)lo >> 32);
    P.step[i][1] = (uint32_t)top;
    P.step[i][2] = (uint32_t)(top >> 32);
  }
}

// rows m_launch.. of the last pair repeat the launch's first row (evaluated,
// never written back)
void fx_shifts(FxBase& P, const double* shifts) {
  for (int kk = 0; kk < kMcMax; ++kk)
    for (int i = 0; i < P.d; ++i) {
      const int src = kk < P.m_launch ? P.k_base + kk : P.k_base;
      P.shift[kk][i] = shift_fixed64(shifts[(size_t)src * P.d + i]);
    }
}

// Launch shape: one resident wave over (point tiles, CTA rows), `rows` rows in the
// largest launch.  max_ctas (> 0) caps the CTAs of one row.
int fx_grid(int occ, uint64_t n, int rows, int max_ctas, int* nblk, int* L, uint64_t* tiles) {
  const int sms = device_sms();
  if (sms <= 0) return fail(QMC_ECUDA, "no CUDA device");
  uint64_t want = std::max<uint64_t>(1, (uint64_t)sms * (uint64_t)std::max(occ, 1) / (uint64_t)rows);
  if (max_ctas > 0) want = std::min<uint64_t>(want, (uint64_t)max_ctas);
  const uint64_t per = (n + want * kThreads - 1) / (want * kThreads);
  *L = (int)std::max<uint64_t>(1, std::min<uint64_t>(per, 512));
  *tiles = (n + (uint64_t)kThreads * *L - 1) / ((uint64_t)kThreads * *L);
  *nblk = (int)std::min<uint64_t>(want, *tiles);
  return QMC_OK;
}

int fx_pairs(int m) { return (std::min(m, kMcMax) + kFxRows - 1) / kFxRows; }

const void* fx_kernel(int d, int tr) {
  switch (d) {
#define QMC_D_CASE(DD) \
  case DD:             \
    return sector_fx_ptr<DD>(tr);
    QMC_D_CASE(1) QMC_D_CASE(2) QMC_D_CASE(3) QMC_D_CASE(4) QMC_D_CASE(5) QMC_D_CASE(6) QMC_D_CASE(7)
    QMC_D_CASE(8)
#undef QMC_D_CASE
    default: return nullptr;
  }
}

}  // namespace

int build_fx_plan(Plan* pl, int32_t d, uint64_t n, int32_t m, const uint64_t* g, const double* shifts,
                  const qmc_transform& t, const qmc_integrand* f, const TuneChoice& tune) {
  // U^-2 F^-1, deg U <= 1, deg F <= 2, d <= 8, no negative coefficient, the
  // constant terms within kFxRange of the coefficient sums
  if (f->kind != QMC_F_SECTOR || f->precision != QMC_FP64 || f->aU != -2 || f->aF != -1 || d > kDFast ||
      tune.force_general || tune.no_fx || tune.L > 0 || (t.kind == QMC_TRANSFORM_KOROBOV && t.alpha != 3) ||
      poly_degree(f->U, d) > 1 || poly_degree(f->F, d) > 2 || !poly_positive(f->U, d) || !poly_positive(f->F, d))
    return QMC_EUNSUPPORTED;
  const std::vector<double> cu = pack_dense(f->U, d, 1), cf = pack_dense(f->F, d, 2);
  int ku = 0, kf = 0;
  double ru = 0.0, rf = 0.0;
  if (!fx_scale(cu, &ku, &ru) || !fx_scale(cf, &kf, &rf)) return QMC_EUNSUPPORTED;
  const int tr = t.kind == QMC_TRANSFORM_KOROBOV ? TR_KOROBOV : (t.kind == QMC_TRANSFORM_BAKER ? TR_BAKER : TR_NONE);
  const void* func = fx_kernel(d, tr);
  if (!func) return QMC_EUNSUPPORTED;

  FxParams base;
  std::memset(&base, 0, sizeof(base));
  base.d = d;
  base.tr = tr;
  fx_lattice(base, n, g);
  base.peaked = tr == TR_KOROBOV && std::max(ru, rf) > kFxPeaked ? 1 : 0;
  // What is added to the constants: what the sums lose on average at z = 0, in
  // their own units.  A dot product drops the fraction of its cross sum (1/2) and per
  // term the last four bits of the coordinate (7.5 of 16 against the coefficient's
  // high word) and the low words' product; a row's product 3/4.  The coordinates are
  // themselves too large by `high` 2^-63 there (truncated products; Korobov's measured
  // on the CPU over s = 1e-6..0.07).
  const double high = tr == TR_KOROBOV ? 6.5 : (tr == TR_BAKER ? -0.5 : -0.25);
  const auto lost = [&](double c, int k, uint32_t ch, uint32_t cl) {
    return 7.5 * std::ldexp((double)ch, -32) + 0.5 * std::ldexp((double)cl, -28) - high * std::ldexp(c, k - 64);
  };
  double more = 0.5;
  for (int i = 0; i < d; ++i) {
    fx_split(cu[1 + i], ku, &base.uh[i], &base.ul[i]);
    more += lost(cu[1 + i], ku, base.uh[i], base.ul[i]);
  }
  base.u0 = fx_fixed(cu[0], ku - 1, more);
  more = 0.0;
  for (int i = 0, off = 1, o = 0; i < d; ++i) {
    const double l = cf[off++];
    double row = 0.5;
    bool any = l != 0.0;
    for (int j = i; j < d; ++j, ++o, ++off) {
      fx_split(cf[off], kf, &base.fh[o], &base.fq[o]);
      if (!(base.fh[o] | base.fq[o])) continue;
      base.fmask[i] |= 2u << (j - i);
      row += lost(cf[off], kf, base.fh[o], base.fq[o]);
      any = true;
    }
    if (!any) continue;
    base.fmask[i] |= 1u;
    base.fl[i] = (uint64_t)std::max<int64_t>(0, (int64_t)fx_fixed(l, kf - 1, row));
    more += 0.75 - high * std::ldexp(l, kf - 65);
  }
  base.f0 = fx_fixed(cf[0], kf - 2, more);
  // value = v 2^(2 su + sf) 2^(2 ku + kf - 252), the smallest shift 2 su + sf
  // taken out; Korobov: v carries 4 more bits, and its weights are (4x(1-x))^3
  // against Eq. (5)'s 140 (x(1-x))^3
  base.value_scale = std::ldexp(1.0, kFxShiftMin + 2 * ku + kf - 252);
  if (tr == TR_KOROBOV) base.value_scale *= std::pow(140.0 / 64.0, (double)d) / 16.0;

  int occ = 0, nblk = 0, L = 0;
  uint64_t tiles = 0;
  // three CTAs of 8 warps saturate an SM's issue slots
  int rc = grid_occupancy(func, 0, tune.occupancy > 0 ? std::min(tune.occupancy, 3) : 3, occ);
  if (rc) return rc;
  pl->grid_rows = fx_pairs(m);
  rc = fx_grid(occ, n, pl->grid_rows, tune.max_ctas, &nblk, &L, &tiles);
  if (rc) return rc;
  pl->param_kind = 5;
  pl->grid_occ = occ;
  pl->grid_capped = true;
  base.L = L;
  base.tiles = tiles;
  base.nblk = nblk;
  pl->nblk = nblk;
  pl->func = func;
  pl->mc = kMcMax;
  pl->final_scale = base.value_scale;
  for (int k0 = 0; k0 < m; k0 += kMcMax) {
    FxParams P = base;
    P.m_launch = std::min(kMcMax, m - k0);
    P.k_base = k0;
    fx_shifts(P, shifts);
    Launch ln;
    ln.func = func;
    ln.grid = dim3(nblk, fx_pairs(P.m_launch));
    ln.params.resize(sizeof(P));
    std::memcpy(ln.params.data(), &P, sizeof(P));
    pl->launches.push_back(std::move(ln));
  }
  return QMC_OK;
}

// largest (sum of U's coefficients) / (its constant), and twice that sum / constant for
// F (y.dF(0) and y.g come one after the other): 1.2e-16 of the estimate
constexpr double kDefFxRange = 250.0;
constexpr double kDefFxMin = 1.0 / 32.0;  // smallest sum of |lambda dF| over the cube
constexpr int kDefFxNode = 55;            // smallest scale of the determinant's nodes: 1.4e-16 of the estimate, at 54 4e-16

// The deformed FAST integrand in fixed point (deformed_fx.cuh) from DefTab's
// constants t (F(0), dF(0), Hessian, half diagonal, minors) and U's cu.
// QMC_EUNSUPPORTED, nothing written, where the scales leave the range in which
// the fixed-point errors stay below the double kernel's.
int build_deformed_fx_plan(Plan* pl, int32_t d, uint64_t n, int32_t m, const uint64_t* g, const double* shifts,
                           const std::vector<double>& t, const std::vector<double>& cu, double lambda,
                           const TuneChoice& tune) {
  if (d > kDefFxMax || !(lambda > 0.0) || tune.L > 0 || tune.no_fx) return QMC_EUNSUPPORTED;
  const void* func = nullptr;
  switch (d) {
    case 1: func = deformed_fx_ptr<1>(); break;
    case 2: func = deformed_fx_ptr<2>(); break;
    case 3: func = deformed_fx_ptr<3>(); break;
    case 4: func = deformed_fx_ptr<4>(); break;
    case 5: func = deformed_fx_ptr<5>(); break;
    case 6: func = deformed_fx_ptr<6>(); break;
  }
  const double* lin = t.data() + 1;
  const double* Hu = lin + d;
  const double* minors = Hu + d * (d + 1) / 2 + d;
  const auto at = [&](int k, int l) {
    const int i = std::min(k, l), j = std::max(k, l);
    return i * d - i * (i - 1) / 2 + (j - i);
  };
  // bounds over the cube: |g'_k|, their sum (y.g'), |m_k|, the recursion's nodes
  double gmax = 0.0, gsum = 0.0, lsum = 0.0, usum = 0.0;
  std::vector<double> growth(d);
  for (int k = 0; k < d; ++k) {
    double gk = std::fabs(lin[k]);
    for (int l = 0; l < d; ++l) gk += std::fabs(Hu[at(k, l)]);
    gk *= lambda;
    gmax = std::max(gmax, gk);
    gsum += gk;
    lsum += std::fabs(lin[k]);
    usum += std::fabs(cu[1 + k]);
    growth[k] = std::hypot(1.0, gk + 0.25 * lambda * std::fabs(Hu[at(k, k)]));
  }
  std::vector<double> node((size_t)1 << d);
  double top = 1.0;
  for (unsigned S = 0; S < (1u << d); ++S) {
    node[S] = std::fabs(minors[S]) * std::pow(lambda, (double)__builtin_popcount(S));
    top = std::max(top, node[S]);
  }
  for (int J = d - 1; J >= 0; --J)
    for (unsigned S = 0; S < (1u << J); ++S) {
      node[S] = growth[J] * node[S] + 0.25 * node[S | (1u << J)];
      top = std::max(top, node[S]);
    }
  // near the origin F and U are their constants, against which the sums' absolute
  // errors count; y.g' gives F in units of lambda
  if (!(std::fabs(t[0]) * kDefFxRange >= lsum + gsum / lambda) || !(std::fabs(cu[0]) * kDefFxRange >= usum) ||
      !(gsum >= kDefFxMin))
    return QMC_EUNSUPPORTED;
  // the largest scale that keeps `most` below 2^bits: g' (and with it m, at most 5/4 of
  // it) and the determinant's nodes (the root carries det J - 1) below 2^62
  const auto scale = [](double most, double bits) { return (int)std::floor(bits - std::log2(std::max(most, 1e-300))); };
  const int cg = std::min({62, scale(gmax, 61.5), scale(gsum, 61.5)});
  const int x = std::min(cg, scale(top + 1.0, 61.9));
  const int cl = std::min(62, scale(lsum, 61.5)), cuq = std::min(62, scale(usum, 61.5));
  if (gmax > 4.0 || 62 - cg > 8 || x < kDefFxNode || cg - x > 8 || cl < 40 || cuq < 40 || !std::isfinite(top) ||
      !std::isfinite(gsum))
    return QMC_EUNSUPPORTED;

  DefFxParams base;
  std::memset(&base, 0, sizeof(base));
  base.d = d;
  base.tr = TR_KOROBOV;
  fx_lattice(base, n, g);
  const auto fixed = [](double c, int q) { return (int64_t)std::llrint(std::ldexp(c, q)); };
  const auto times = [&](double a, double b, int q) {  // a b without the product's rounding
    const double hi = a * b;
    return fixed(hi, q) + fixed(std::fma(a, b, -hi), q);
  };
  const auto limb = [](int64_t v) {  // to the nearest, the last three bits are dropped
    return FxLimb{(int32_t)((v + 4) >> 31), (int32_t)(((uint32_t)(v + 4) >> 3) & 0x0FFFFFFFu)};
  };
  for (int k = 0; k < d; ++k) {
    for (int l = k; l < d; ++l) base.H[at(k, l)] = limb(times(-lambda, Hu[at(k, l)], cg));
    base.Q[k] = limb(times(-0.5 * lambda, Hu[at(k, k)], cg));
    base.gl[k] = times(-lambda, lin[k], cg) + 4;
    base.fl[k] = limb(fixed(lin[k], cl));
    base.u[k] = limb(fixed(cu[1 + k], cuq));
  }
  for (unsigned S = 0; S < (1u << d); ++S) {
    const double h = minors[S] * std::pow(-lambda, (double)__builtin_popcount(S));
    base.hs[S] = fixed(h, x);
    base.hl[S] = limb(base.hs[S]);
    base.hs[S] += 4;
  }
  base.sh = 62 - cg;
  base.mx = cg - x;
  base.half = 1 << (27 - base.sh);
  base.four = 1 << (30 - base.sh);
  base.around = ((1 << base.sh) >> 1) - 4 + (4 << base.sh);  // and 4 more for its own limbs
  base.mround = ((1 << base.mx) >> 1) - 4;
  base.has_lin = lsum > 0.0;
  base.u0 = cu[0];
  base.su = std::ldexp(1.0, -cuq);
  base.f0 = t[0];
  base.c1 = std::ldexp(0.5, -cl);
  base.c2 = -std::ldexp(0.5, -cg) / lambda;
  base.c3 = std::ldexp(1.0, -cg) / lambda;
  base.sd = std::ldexp(1.0, -x);
  base.value_scale = korobov_scale(kKorCentred, d) * 0x1p-192;

  int occ = 0, nblk = 0, L = 0;
  uint64_t tiles = 0;
  int rc = grid_occupancy(func, 0, tune.occupancy, occ);
  if (rc) return rc;
  pl->grid_rows = std::min(m, kMcMax);
  rc = fx_grid(occ, n, pl->grid_rows, 0, &nblk, &L, &tiles);
  if (rc) return rc;
  pl->param_kind = 5;
  pl->grid_occ = occ;
  pl->grid_capped = false;  // as the other deformed plans
  base.L = L;
  base.tiles = tiles;
  base.nblk = nblk;
  pl->nblk = nblk;
  pl->func = func;
  pl->mc = kMcMax;
  pl->final_scale = base.value_scale;
  pl->is_complex = 1;
  for (int k0 = 0; k0 < m; k0 += kMcMax) {
    DefFxParams P = base;
    P.m_launch = std::min(kMcMax, m - k0);
    P.k_base = k0;
    fx_shifts(P, shifts);
    Launch ln;
    ln.func = func;
    ln.grid = dim3(nblk, P.m_launch);
    ln.params.resize(sizeof(P));
    std::memcpy(ln.params.data(), &P, sizeof(P));
    pl->launches.push_back(std::move(ln));
  }
  return QMC_OK;
}

int fx_rebase(Plan* pl, uint64_t n, const uint64_t* g, int max_ctas) {
  int nblk = 0, L = 0;
  uint64_t tiles = 0;
  int rc = fx_grid(pl->grid_occ, n, pl->grid_rows, pl->grid_capped ? max_ctas : 0, &nblk, &L, &tiles);
  if (rc) return rc;
  for (Launch& ln : pl->launches) {
    FxBase& P = *reinterpret_cast<FxBase*>(ln.params.data());
    fx_lattice(P, n, g);
    P.L = L;
    P.tiles = tiles;
    P.nblk = nblk;
    ln.grid.x = nblk;
  }
  pl->n = n;
  pl->nblk = nblk;
  pl->tune.max_ctas = max_ctas;
  return QMC_OK;
}

void fx_reshift(Plan* pl, const double* shifts) {
  for (Launch& ln : pl->launches) fx_shifts(*reinterpret_cast<FxBase*>(ln.params.data()), shifts);
}

}  // namespace qmc
