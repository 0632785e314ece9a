// Plan builder for contour-deformed (complex) sector integrands.
#include <algorithm>
#include <cmath>
#include <cstdlib>
#include <cstring>

#include "deformed.cuh"
#include "plan.h"

namespace qmc {

// QMC_DEFORMED_PACKED=0 keeps FP32 plans on the one-shift kernel.
static bool deformed_packed_enabled() {
  const char* e = std::getenv("QMC_DEFORMED_PACKED");
  return !(e && e[0] == '0');
}

// The packed FP32 variant (two shifts per instruction), d <= kDef2DMax.
static const void* deformed2_ptr(int d) {
  switch (d) {
    case 1: return (const void*)&deformed2_kernel<1>;
    case 2: return (const void*)&deformed2_kernel<2>;
    case 3: return (const void*)&deformed2_kernel<3>;
    case 4: return (const void*)&deformed2_kernel<4>;
    case 5: return (const void*)&deformed2_kernel<5>;
    default: return nullptr;
  }
}

// det(H_off restricted to rows S and columns cols) by expansion along its first row.
// seen (2^2d) keeps the minors found for the other subsets of one table: d = 7, all
// 128 principal minors, 194 -> 23 us.
static double minor_off(const std::vector<double>& H, int d, unsigned S, unsigned cols, std::vector<double>& seen) {
  if (!S) return 1.0;
  double& known = seen[(size_t)S << d | cols];
  if (!std::isnan(known)) return known;
  int r = 0;
  while (!(S >> r & 1u)) ++r;
  double det = 0.0, sign = 1.0;
  for (int c = 0; c < d; ++c) {
    if (!(cols >> c & 1u)) continue;
    if (c != r && H[(size_t)r * d + c] != 0.0)
      det += sign * H[(size_t)r * d + c] * minor_off(H, d, S & ~(1u << r), cols & ~(1u << c), seen);
    sign = -sign;
  }
  return known = det;
}

// DefTab's constants.
static std::vector<double> fast_table(const std::vector<double>& cf, int d, double lambda) {
  std::vector<double> H((size_t)d * d, 0.0), t;
  t.push_back(cf[0]);
  for (int k = 0, off = 1; k < d; ++k) {
    t.push_back(cf[off++]);
    for (int l = k; l < d; ++l, ++off) H[(size_t)k * d + l] = H[(size_t)l * d + k] = (k == l ? 2.0 : 1.0) * cf[off];
  }
  for (int k = 0; k < d; ++k)
    for (int l = k; l < d; ++l) t.push_back(H[(size_t)k * d + l]);
  for (int k = 0; k < d; ++k) t.push_back(0.5 * H[(size_t)k * d + k]);
  std::vector<double> seen((size_t)1 << 2 * d, std::nan(""));
  for (unsigned S = 0; S < (1u << d); ++S) t.push_back(minor_off(H, d, S, S, seen));
  for (double v : {lambda, -lambda, 2.0 * lambda, 0.5}) t.push_back(v);
  return t;
}

// Offset of q_ij (i <= j) in the nested degree-2 layout (host copy of q_off).
static int q_off_host(int D, int i, int j) {
  int off = 1;
  for (int a = 0; a < i; ++a) off += 1 + (D - a);
  return off + 1 + (j - i);
}

template <typename R>
static int build_def(Plan* pl, int32_t d, uint64_t n, int32_t m, const uint64_t* g, const double* shifts,
                     const qmc_transform& t, const qmc_integrand* f, const TuneChoice& tune) {
  if (d > kDFast) return fail(QMC_EUNSUPPORTED, "deformed sector integrands need d <= %d", kDFast);
  RuleParams<R> base;
  fill_common(base, d, n, g, t, f);
  auto cf = pack_dense(f->F, d, 2);
  // J = I + i M with M_kl = -lam (y_k (1 - y_k) S_kl + delta_kl (1 - 2 y_k) dF_k), S = Hessian of F.
  // |J_kk| >= 1 and sum_{l != k} |M_kl| <= lam / 4 * sum_{l != k} |S_kl|: below 1 for every row,
  // J is strictly row diagonally dominant on the whole cube and LU needs no pivoting.
  double worst = 0.0;
  for (int k = 0; k < d; ++k) {
    double row = 0.0;
    for (int l = 0; l < d; ++l) {
      if (l == k) continue;
      const int a = k < l ? k : l, b = k < l ? l : k;
      row += std::fabs(cf[q_off_host(d, a, b)]);
    }
    worst = std::max(worst, 0.25 * f->lambda * row);
  }
  const bool fast = worst < 1.0 && t.kind == QMC_TRANSFORM_KOROBOV && t.alpha == 3 && !tune.force_general;
  const bool u_linear = poly_degree(f->U, d) <= 1;  // U on its degree-1 slots only
  // FP32 with two shifts per instruction: the FAST variant, U^-2 F^-1, d <= kDef2DMax
  const bool packed = sizeof(R) == 4 && fast && u_linear && d <= kDef2DMax && f->aU == -2 && f->aF == -1 &&
                      deformed_packed_enabled();
  const void* func = nullptr;
  switch (d) {
#define QMC_D_CASE(DD) \
  case DD:             \
    func = deformed_ptr<R, DD>(fast, u_linear); \
    break;
    QMC_D_CASE(1) QMC_D_CASE(2) QMC_D_CASE(3) QMC_D_CASE(4) QMC_D_CASE(5) QMC_D_CASE(6) QMC_D_CASE(7)
    QMC_D_CASE(8)
#undef QMC_D_CASE
    default: break;
  }
  if (packed) func = deformed2_ptr(d);
  // FP64 FAST: a CTA row per shift row, det J from the minors' table
  const bool rows64 = sizeof(R) == 8 && fast && d <= kDefFastMax;
  if (rows64 && u_linear && f->aU == -2 && f->aF == -1) {
    int rc = build_deformed_fx_plan(pl, d, n, m, g, shifts, fast_table(cf, d, f->lambda), pack_dense(f->U, d, 1),
                                    f->lambda, tune);
    if (rc != QMC_EUNSUPPORTED) return rc;
  }
  if (!func) return fail(QMC_EUNSUPPORTED, "no deformed kernel for d=%d", d);
  auto cu = pack_dense(f->U, d, u_linear ? 1 : 2);
  for (size_t i = 0; i < cu.size(); ++i) base.cU[i] = (R)cu[i];
  if (rows64) {
    const std::vector<double> t = fast_table(cf, d, f->lambda);
    static_assert(DefTab<kDefFastMax>::END <= kPolyCoefMax, "deformed constants");
    for (size_t i = 0; i < t.size(); ++i) base.cF[i] = (R)t[i];
  } else {
    for (size_t i = 0; i < cf.size(); ++i) base.cF[i] = (R)cf[i];
    for (int k = 0; k < d; ++k)  // -lambda d2F/dy_k dy_l (constant: F has degree 2)
      for (int l = 0; l < d; ++l) {
        const int a = k < l ? k : l, b = k < l ? l : k;
        const double h = (k == l ? 2.0 : 1.0) * cf[q_off_host(d, a, b)];
        base.cF[kDefHessOff + k * d + l] = (R)(-f->lambda * h);
      }
  }
  if (packed) {  // (c, c) pairs: U's linear slots, F's slots, then the Hessian of F, k-major
    int o = 0;
    for (double v : cu) base.cp[o++] = make_float2((float)v, (float)v);
    for (double v : cf) base.cp[o++] = make_float2((float)v, (float)v);
    for (int k = 0; k < d; ++k)
      for (int l = 0; l < d; ++l) {
        const float h = (float)((k == l ? 2.0 : 1.0) * cf[q_off_host(d, std::min(k, l), std::max(k, l))]);
        base.cp[o++] = make_float2(h, h);
      }
    static_assert(1 + kDef2DMax + poly_slots(kDef2DMax, 2) + kDef2DMax * kDef2DMax <= kPairCoefMax, "coefficient pairs");
  }
  // Transform weight constants.  FP64 normalises each factor in the general
  // kernel; its FAST kernel cubes the product of 4x(1-x) in units of 2^-64.
  // FP32 FAST multiplies the factors u and cubes the product: (2a+1)!/(a!)^2
  // = 140 per dimension remains; other FP32 Korobov plans raise the product of
  // the factors 4u to the power alpha: ((2a+1)!/(a!)^2 / 4^a) per dimension.
  base.value_scale = 1.0;
  if (fast && sizeof(R) == 8) base.value_scale = korobov_scale(kKorCentred, d) * 0x1p-192;
  else if (sizeof(R) == 4 && base.tr == TR_KOROBOV)
    base.value_scale = fast ? korobov_scale(3, d)
                            : std::pow((double)base.kor[7] / std::pow(4.0, (double)base.alpha), (double)d);
  base.check_finite = 1;
  int nblk = 0, L = 0, occ = 0;
  uint64_t tiles = 0;
  int rc = grid_occupancy(func, 0, tune.occupancy, occ);
  if (rc) return rc;
  const int mc = rows64 ? kMcMax : kMcDeformed;  // the others: as many as they have shared accumulators
  pl->grid_rows = rows64 ? std::min(m, kMcMax) : 1;
  rc = grid_shape(occ, n, rows_cap(pl, occ, 0), tune.L, nblk, L, tiles);
  if (rc) return rc;
  pl->param_kind = sizeof(R) == 4 ? 1 : 2;
  pl->grid_occ = occ;
  pl->grid_capped = false;  // one resident wave whatever the caller's cap
  base.L = L;
  base.tiles = tiles;
  base.nblk = nblk;
  pl->nblk = nblk;
  pl->func = func;
  pl->mc = mc;
  pl->final_scale = base.value_scale;
  pl->is_complex = 1;
  for (int k0 = 0; k0 < m; k0 += mc) {
    const int mk = std::min(mc, m - k0);
    RuleParams<R> P = base;
    P.m_launch = mk;
    P.k_base = k0;
    for (int kk = 0; kk < mc; ++kk)  // rows mk.. repeat row k0 (evaluated at most, never written back)
      for (int i = 0; i < d; ++i)
        set_shift(P, kk, i, shift_fixed64(shifts[(size_t)(kk < mk ? k0 + kk : k0) * d + i]));
    Launch ln;
    ln.func = func;
    ln.grid = dim3(nblk, rows64 ? mk : 1);
    ln.params.resize(sizeof(P));
    std::memcpy(ln.params.data(), &P, sizeof(P));
    pl->launches.push_back(std::move(ln));
  }
  return QMC_OK;
}

int build_deformed_plan(Plan* pl, int32_t d, uint64_t n, int32_t m, const uint64_t* g, const double* shifts,
                        const qmc_transform& t, const qmc_integrand* f, const TuneChoice& tune) {
  if (f->precision == QMC_FP32EVAL) return build_def<float>(pl, d, n, m, g, shifts, t, f, tune);
  return build_def<double>(pl, d, n, m, g, shifts, t, f, tune);
}

}  // namespace qmc
