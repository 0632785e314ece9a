// The FP64 FAST contour integrand in signed 64-bit fixed point.
//
// What bounds the double kernel (deformed64_kernel): the FP64 pipe, 225 operations
// a value at d = 5, 64 issue slots each.  A product of two 62-bit numbers takes
// three 32x32 -> 64-bit multiply-adds, 12 slots, so the gradient, the contour, the
// quadratic forms and the determinant's recursion (def_fast's formulas, all of
// bounded size) run in integers; U, F and det J - 1 are then converted, and U^-2
// F^-1 det J, whose size is not bounded, is formed in double: about 40 FP64
// operations, which run beside the integer ones.
//
// Measured (GB300, d = 5, n = 262139, m = 20): 2.26 -> 0.70 ms (0.68 with limbs and
// sums truncated instead of rounded); in that form d = 2..4 took 0.48 to 0.51 ms, d = 6
// 1.12 ms (double kernels with LU 1.5 to 3.6 and 6.4 ms).  What bounds it: issue
// slots at d = 5 (568 multiply-adds of four and 1750 others a value, 78 % of the slots),
// the FP64 pipe below.  Two CTAs per SM at 128 registers with 36 spilled bytes (d = 5);
// one CTA at 156 registers took 1.5 times as long.
//
// Numbers.  An int64 X stands for X 2^-q, |X| < 2^62, and is multiplied by its limbs
// h = X >> 31 and l = (X >> 3) mod 2^28:
//   X Y / 2^62 = h h' + (h l' + l h') / 2^28,
// the cross products short enough (2^59) that the sums of a dot product share one
// 64-bit accumulator.  The last three bits (rounded) and l l' (its mean put back) are
// dropped, 2^-58 of the full range at most.  Scales per plan, from bounds over the cube (fixed64.cu): cg for
// g' = -lambda dF, v = y (1 - y) g', m = y (1 - y) H'_kk + (1 - 2y) g' and the
// quadratic forms, x for the recursion's nodes.  A product with a Q(cg) number comes
// out 62 - cg = sh bits low; the sum is shifted back before its low part is added.
// Error against 80-bit floats, d = 1..6, lambda 0.02 to 0.4, constants down to 1/120
// of the coefficients' sum: an estimate 1e-18 to 1.2e-16 (root mean square of eight
// integrands), a value 3e-16 to 5e-15 over the cube; more where Re F crosses zero and
// |F| is small (d = 2, lambda <= 0.05: 4e-16 and 3e-13).  With truncated limbs and sums and one bit less an
// estimate was up to 2.4e-15 off, the determinant's truncations being multiplied up
// its recursion.
#pragma once

#include "deformed.cuh"

namespace qmc {

__device__ __forceinline__ int64_t fx_mads(int32_t a, int32_t b, int64_t c) {
  int64_t r;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
  return r;
}

__device__ __forceinline__ FxLimb fx_limb(int64_t X) {
  return {(int32_t)(X >> 31), (int32_t)(((uint32_t)X >> 3) & 0x0FFFFFFFu)};
}

// A sum of n products, shifted left by sh at the end: the cross sum starts with half
// a unit, half = 2^(27 - sh), and with what the n products of low limbs amount to on
// average (2^54 each), so that nothing is lost on average.
// Results that are taken apart into limbs carry four units more, which rounds the
// limbs' three dropped bits: from their sum's start (r, or four = 4 2^(28 - sh) in the
// cross sum), and in the determinant's recursion from its leaves on (x' = x + 4
// keeps through x - re and x + im), until the root takes them off.
struct FxProd {
  int64_t r, c;
  __device__ __forceinline__ explicit FxProd(int n, int32_t start = 1 << 27, int64_t r0 = 0)
      : r(r0), c(start + (n << 26)) {}
  __device__ __forceinline__ void add(const FxLimb& a, const FxLimb& b) {
    r = fx_mads(a.h, b.h, r);
    c = fx_mads(a.h, b.l, c);
    c = fx_mads(a.l, b.h, c);
  }
  __device__ __forceinline__ int64_t value() const { return r + (c >> 28); }
  __device__ __forceinline__ int64_t value(int sh) const { return (int64_t)((uint64_t)r << sh) + (c >> (28 - sh)); }
};

struct FxCx {
  int64_t re, im;
};

// def_node and def_root in fixed point: ml, al the limbs of m and of y (1 - y) in
// Q(cg), nodes in Q(x).
template <int D, int J, int S>
__device__ __forceinline__ FxCx defx_node(const DefFxParams& P, const FxLimb* ml, const FxLimb* al) {
  if constexpr (J == D - 1) {
    FxProd p((S & (S - 1)) != 0 ? 2 : 1, P.half + P.four);
    if constexpr ((S & (S - 1)) != 0) p.add(ml[J], P.hl[S]);
    p.add(al[J], P.hl[S | (1 << J)]);
    return {(S & (S - 1)) != 0 ? P.hs[S] : 0, p.value(P.sh)};
  } else {
    const FxCx x = defx_node<D, J + 1, S>(P, ml, al), y = defx_node<D, J + 1, S | (1 << J)>(P, ml, al);
    constexpr bool kRe = J < D - 2 || (S & (S - 1)) != 0;  // else x.re = 0
    FxProd re(2, kRe ? P.half : P.half - P.four), im(kRe ? 2 : 1, P.half);
    re.add(ml[J], fx_limb(x.im));
    re.add(al[J], fx_limb(y.im));
    if constexpr (kRe) im.add(ml[J], fx_limb(x.re));
    im.add(al[J], fx_limb(y.re));
    return {x.re - re.value(P.sh), x.im + im.value(P.sh)};
  }
}

template <int D, int J>
__device__ __forceinline__ FxCx defx_root(const DefFxParams& P, const int64_t* m, const FxLimb* ml, const FxLimb* al) {
  if constexpr (J == D - 1) {
    return {0, ((m[J] + P.mround) >> P.mx) + 4};
  } else {
    const FxCx x = defx_root<D, J + 1>(P, m, ml, al), y = defx_node<D, J + 1, 1 << J>(P, ml, al);
    FxProd re(2, J < D - 2 ? P.half : P.half - P.four), im(J < D - 2 ? 2 : 1, P.half);
    re.add(ml[J], fx_limb(x.im));
    re.add(al[J], fx_limb(y.im));
    if constexpr (J < D - 2) im.add(ml[J], fx_limb(x.re));
    im.add(al[J], fx_limb(y.re));
    return {x.re - re.value(P.sh), ((m[J] + P.mround) >> P.mx) + x.im + im.value(P.sh)};
  }
}

template <int D, bool TERM>
__device__ __forceinline__ Cx<double> deformed_fx_value(const DefFxParams& P, const uint64_t* base,
                                                        const uint64_t* shift) {
  using T = DefTab<D>;
  const auto H = [&](int k, int l) { return P.H[T::h(k, l) - T::H]; };
  FxLimb y[D];
  double wt = 1.0;
  uint64_t wf = 0;
#pragma unroll
  for (int i = 0; i < D; ++i) {
    uint64_t u;
    const uint64_t z = fx_coord<TR_KOROBOV>(base[i] + shift[i], u);
    if constexpr (TERM) wt *= __ull2double_rn(u) * (i == 0 ? 1.0 : 0x1p-64);
    else wf = i == 0 ? u : fx_mulhi_add(wf, u, 0);
    y[i] = {(int32_t)(z >> 32), (int32_t)((uint32_t)z >> 4)};  // z / 2 in Q62
  }
  if constexpr (!TERM) wt = __ull2double_rn(wf);
  wt = wt * wt * wt;
  int64_t m[D];
  FxLimb ml[D], al[D], vl[D];
  FxProd ur(D), ui(D, P.half), yl(D), yg(D), vg(D, P.half), vr(D, P.half);
#pragma unroll
  for (int k = 0; k < D; ++k) {
    FxProd p(D);
#pragma unroll
    for (int l = 0; l < D; ++l) p.add(H(k, l), y[l]);
    const int64_t gk = P.gl[k] + p.value();
    const FxLimb g = fx_limb(gk);
    FxProd q(1, 1 << 27, 4);
    q.add(y[k], FxLimb{0x7FFFFFFF - y[k].h, 0x0FFFFFFF - y[k].l});
    const int64_t a = q.value();  // y (1 - y), Q62
    const FxLimb af = fx_limb(a);
    FxProd v(1, 1 << 27, 4);
    v.add(af, g);
    vl[k] = fx_limb(v.value());
    // 1 - 2y in Q62 from y's limbs: (2^31 - 1 - 2h, 2^28 - 1 - 2l) with l's carry
    const int32_t wl = 0x0FFFFFFF - 2 * y[k].l;
    const FxLimb w = {(int32_t)(0x7FFFFFFFu - 2u * (uint32_t)y[k].h + (uint32_t)(wl >> 28)), wl & 0x0FFFFFFF};
    FxProd d(2, 1 << 27, 4);
    d.add(af, H(k, k));
    d.add(w, g);
    m[k] = d.value();
    ml[k] = fx_limb(m[k]);
    al[k] = fx_limb((a + P.around) >> P.sh);
    ur.add(P.u[k], y[k]);
    ui.add(P.u[k], vl[k]);
    yg.add(y[k], g);
    vg.add(vl[k], g);
    if (P.has_lin) yl.add(P.fl[k], y[k]);
  }
#pragma unroll
  for (int k = 0; k < D; ++k) {
    FxProd r(D - k, P.half + P.four);
    r.add(P.Q[k], vl[k]);
#pragma unroll
    for (int l = k + 1; l < D; ++l) r.add(H(k, l), vl[l]);
    vr.add(vl[k], fx_limb(r.value(P.sh)));
  }
  const FxCx del = defx_root<D, 0>(P, m, ml, al);
  const auto dbl = [](int64_t X) { return __ll2double_rn(X); };
  const Cx<double> U{fma_(dbl(ur.value()), P.su, P.u0), dbl(ui.value(P.sh)) * P.su};
  double fr = fma_(dbl(yg.value()), P.c2, P.f0);
  if (P.has_lin) fr = fma_(dbl(yl.value()), P.c1, fr);
  fr = fma_(dbl(vr.value(P.sh)), P.c3, fr);
  const int64_t fi = vg.value(P.sh);  // v.g' = sum y (1 - y) g'^2 >= 0
  const Cx<double> F{fr, dbl(fi > 0 ? fi : 0) * -P.c3};
  const Cx<double> dm1{dbl(del.re - (D > 1 ? 4 : 0)) * P.sd, dbl(del.im - 4) * P.sd};
  const Cx<double> rv = crecip(cmul(cmul(U, U), F));
  const Cx<double> t = cmul(dm1, rv);
  return {(rv.re + t.re) * wt, (rv.im + t.im) * wt};
}

// One shift row per CTA row, a thread's points kThreads apart.  Im F(w) <= 0 by
// construction (F is quadratic), so no point is counted as on the wrong side.
template <int D>
__global__ void __launch_bounds__(kThreads, 2)
    deformed_fx_kernel(const __grid_constant__ DefFxParams P, double* __restrict__ partial,
                       unsigned long long* __restrict__ counters, const SampleIO sio) {
  if (sio.count > 0) {
    int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= sio.count) return;
    const uint64_t j = sio.j[s];
    const int k = sio.k[s];
    uint64_t base[D], sh[D];
#pragma unroll
    for (int i = 0; i < D; ++i) {
      const uint32_t idx = lattice_index(j, P.g[i], P.n);
      base[i] = frac64(idx, P.rc);
      sh[i] = P.shift[k][i];
      if (sio.idx) sio.idx[(size_t)s * D + i] = idx;
      if (sio.coord) sio.coord[(size_t)s * D + i] = coord_used<double>(base[i] + sh[i]);
    }
    const Cx<double> v = deformed_fx_value<D, true>(P, base, sh);
    sio.values[2 * (size_t)s] = v.re * P.value_scale;
    sio.values[2 * (size_t)s + 1] = v.im * P.value_scale;
    return;
  }
  const int k = blockIdx.y;
  uint64_t sh[D];
#pragma unroll
  for (int i = 0; i < D; ++i) sh[i] = P.shift[k][i];
  double re = 0.0, im = 0.0;
  unsigned nbad = 0;
  const uint64_t tile_pts = (uint64_t)kThreads * (uint64_t)P.L;
  for (uint64_t tile = blockIdx.x; tile < P.tiles; tile += gridDim.x) {
    const uint64_t j0 = tile * tile_pts + threadIdx.x;
    if (j0 >= P.n) continue;
    const uint64_t left = (P.n - j0 + kThreads - 1) / kThreads;
    const int steps = left < (uint64_t)P.L ? (int)left : P.L;
    FxWalk96<D> walk;
    walk.start(P, j0);
#pragma unroll 1
    for (int s = 0; s < steps; ++s) {
      const Cx<double> v = deformed_fx_value<D, false>(P, walk.base, sh);
      const bool ok = finite_(v.re) && finite_(v.im);
      nbad += ok ? 0u : 1u;
      re += ok ? v.re : 0.0;
      im += ok ? v.im : 0.0;
      walk.step(P);
    }
  }
  block_sum2(re, im, nbad, 0u, counters, partial + ((size_t)(P.k_base + k) * P.nblk + blockIdx.x) * 2);
}

}  // namespace qmc
