// FP64 rule of the separable integrands (constant, separable exponential,
// cosine), runtime d.
//
// What bounds it.  The FP64 pipe: 2 operations per SM and clock, so a warp
// instruction holds it for 16 clocks.  Coordinates and the Korobov-3 weight
// therefore come from 64-bit fixed point (fx_coord), which leaves per dimension one
// conversion and the integrand's own three operations: d = 3 takes about 35
// FP64 operations a value with the exponential, against 75 with the transform in
// double.  Weights other than 3 keep the double transform, and so do exponents and
// factors above kSepFixedMax: near 0 the double transform's coordinate is accurate
// relative to itself, the fixed-point one to about 2 units of 2^-63.
//
// Layout.  One shift row per CTA row, a thread's points kThreads apart: a
// value is worth some 600 clocks of the pipe to a warp, so sharing a point between
// shifts saves nothing, and a small rule (n = 10007, m = 10) spreads over
// the chip instead of giving 40 CTAs eight shifts each, one launch after the
// other.  That call: 128 -> 73 us.
#pragma once

#include "fixed64.cuh"

namespace qmc {

template <int TR, bool KOR3, int FK>  // KOR3: weight 3 in fixed point
struct Sep64 {
  // TERM: a single listed term, its weight to full relative precision
  template <bool TERM, class BASE>
  static __device__ __forceinline__ double value(const RuleParams<double>& P, int k, BASE base) {
    double w = 1.0, prod = 1.0, lin = 0.0;
    uint64_t wf = ~0ull;
    int ew = 0;
#pragma unroll 1
    for (int i = 0; i < P.d; ++i) {
      const uint64_t X = base(i) + P.shift64[k][i];
      double z;  // fixed-point coordinates: 2^63 z, the power of two is in sep_c and sep_b
      if constexpr (TR == TR_KOROBOV && !KOR3) {
        z = coord_f64<TR, 0>(X, P.kor, P.alpha, w);
      } else {
        uint64_t u = 0, zf;
        if constexpr (TR == TR_KOROBOV) {
          zf = fx_coord_centred(X, u);
          if constexpr (TERM) {
            w *= __ull2double_rn(u) * 0x1p-64;
          } else {  // normalised: of 16 factors only 2^-14 may be left, less where the integrand peaks
            wf = i == 0 ? u : fx_mulhi_add(wf, u, 0);
            const int s = fx_clz64(wf);
            wf <<= s;
            ew += s;
          }
        } else {
          zf = fx_coord<TR>(X, u);
        }
        if constexpr (FK != FK_CONST) z = __ull2double_rn(zf);
      }
      if constexpr (FK == FK_SEPEXP) {
        prod *= fma_(P.sep_c[i], z, 1.0);
        lin = fma_(P.sep_b[i], z, lin);
      } else if constexpr (FK == FK_TRIG) {
        lin = fma_(P.sep_c[i], z, lin);
      }
    }
    double v = 1.0;
    if constexpr (FK == FK_SEPEXP) v = prod * exp(lin);
    else if constexpr (FK == FK_TRIG) v = cospi(2.0 * lin);
    if constexpr (TR == TR_KOROBOV) {
      if constexpr (KOR3) {
        if constexpr (!TERM) w = __ull2double_rn(wf) * 0x1p-64;
        w = w * w * w;
        if constexpr (!TERM) w *= 3 * ew < 1000 ? __longlong_as_double((long long)(1023 - 3 * ew) << 52) : 0.0;
      }
      v *= w;
    }
    return v;
  }
};

template <int TR, bool KOR3, int FK>
__global__ void __launch_bounds__(kThreads)
    separable64_kernel(const __grid_constant__ RuleParams<double> P, double* __restrict__ partial,
                       unsigned long long* __restrict__ counters, const SampleIO sio) {
  using S = Sep64<TR, KOR3, FK>;
  if (sio.count > 0) {
    int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= sio.count) return;
    const uint64_t j = sio.j[s];
    const int k = sio.k[s];
    for (int i = 0; i < P.d; ++i) {
      const uint32_t idx = lattice_index(j, P.g[i], P.n);
      if (sio.idx) sio.idx[(size_t)s * P.d + i] = idx;
      if (sio.coord) sio.coord[(size_t)s * P.d + i] = coord_used<double>(frac64(idx, P.rc) + P.shift64[k][i]);
    }
    const double v =
        S::template value<true>(P, k, [&](int i) { return frac64(lattice_index(j, P.g[i], P.n), P.rc); });
    sio.values[2 * (size_t)s] = v * P.value_scale;
    sio.values[2 * (size_t)s + 1] = 0.0;
    return;
  }
  // g_i / n to 128 bits: the fraction of a point is j times it, modulo 1
  __shared__ Recip gf[QMC_DMAX];
  __shared__ double red[kThreads];
  if (threadIdx.x < P.d) {
    const uint64_t g = P.g[threadIdx.x];
    gf[threadIdx.x] = Recip{g * P.rc.rhi + __umul64hi(g, P.rc.rlo), g * P.rc.rlo};
  }
  __syncthreads();
  const int k = blockIdx.y;
  double sum = 0.0;
  unsigned nbad = 0;
  const uint64_t tile_pts = (uint64_t)kThreads * (uint64_t)P.L;
  for (uint64_t tile = blockIdx.x; tile < P.tiles; tile += gridDim.x) {
    const uint64_t j0 = tile * tile_pts + threadIdx.x;
    if (j0 >= P.n) continue;
    const uint64_t left = (P.n - j0 + kThreads - 1) / kThreads;
    const int steps = left < (uint64_t)P.L ? (int)left : P.L;
#pragma unroll 1
    for (int s = 0; s < steps; ++s) {
      const uint32_t j = (uint32_t)j0 + (uint32_t)s * kThreads;
      double v = S::template value<false>(P, k, [&](int i) { return frac64(j, gf[i]); });
      if (P.check_finite) {
        const bool ok = finite_(v);
        nbad += ok ? 0u : 1u;
        v = ok ? v : 0.0;
      }
      sum += v;
    }
  }
  // fixed-order sum: a lane of warp 0 adds eight threads' sums, then the warp tree
  red[threadIdx.x] = sum;
  const unsigned long long bad = warp_sum_u64((unsigned long long)nbad);
  if ((threadIdx.x & 31) == 0 && bad) atomicAdd(&counters[0], bad);
  __syncthreads();
  if (threadIdx.x < 32) {
    double t = red[threadIdx.x];
#pragma unroll
    for (int w = 1; w < kThreads / 32; ++w) t += red[threadIdx.x + 32 * w];
    t = warp_sum_d(t);
    if (threadIdx.x == 0) {
      const size_t slot = ((size_t)(P.k_base + k) * P.nblk + blockIdx.x) * 2;
      partial[slot] = t;
      partial[slot + 1] = 0.0;
    }
  }
}

}  // namespace qmc
