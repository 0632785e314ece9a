// FP64 sector rule in 64-bit fixed point (integer pipes).
//
// What bounds it.  This part issues 2 FP64 operations per SM and clock, and a
// sector value under FP64 takes 39 (d = 6, baker) to 170 (d = 8, Korobov 3) of
// them: the double kernels sat on that pipe.  A 32x32 -> 64-bit multiply-add
// runs at 32 per SM and clock (four issue slots of 128), three of them make a
// 64-bit high product, so the whole value is evaluated in integers: coordinates, U, F, the reciprocal, the
// transform weight and the sum.  No FP64 instruction is left in the loop.
//
// Formats (unsigned fractions; Qk holds x 2^k).  Coordinates z are Q63.  The
// coefficients of U and F are scaled by 2^k so that their sum stays below
// 2^64; every product takes the high 64 bits, so a chain of products steps down
// by one bit: U's terms Qk -> U in Q(k-1) < 2^63, F's quadratic terms Qk -> rows
// Q(k-1) -> F in Q(k-2) < 2^62.  U and F are then normalised to [2^63, 2^64) by
// their leading zeros, which keeps U^2 F and its reciprocal to ~2^-56 relative.
// The value re-enters fixed point as V 2^t (t <= 30) and is summed exactly in
// 128 bits.
//
// Precision.  With R the larger (coefficient sum) / (constant term) of U and F, a
// unit of U is R 2^-63 of its smallest value and one of F R 2^-62.  What the dropped
// products and the coordinates' truncations take away is 4 to 10 units with a spread
// of 2 to 3; its mean at the corner z = 0, where U and F are smallest and such
// integrands peak, goes into the constants (fixed64.cu), so that the spread
// averages out in a sum and half a unit of rounding is left.  The Korobov weight is a product of
// factors in Q64, whose steps count where the integrand peaks where the weight is
// small: from R = kFxPeaked on it is carried normalised.  The host admits R up to
// kFxRange.  Evaluated on the CPU against 80-bit floats (8 integrands of 400000
// points each per d, transform and R), relative error of the estimate and of a
// value (root mean square):
//             d   R      here              double chain
//   Korobov   1   64     1.3e-17 1.3e-16   2.2e-18 1.3e-15
//             1   1000   1.5e-16 2.9e-15   6.9e-18 3.7e-15
//             8   64     3.0e-17 2.7e-15   7.5e-18 5.0e-15
//             8   1000   1.4e-18 4.2e-17   5.7e-18 5.3e-15
//   baker     1   64     4.2e-18 3.5e-16   9.9e-17 5.7e-14
//             1   1000   1.1e-16 2.2e-14   4.2e-15 3.6e-12
// (the double chain's baker and untransformed coordinates are multiples of 2^-53 and
// 2^-52; its sums' own rounding is not in the figures).  With the mean taken over the
// whole cube, one bit less and the weight never normalised, R = 1000 left 1.5e-15 of
// the estimate at d = 1 and 1e-15 (6e-13 of a value) at d = 8.
//
// Measured (GB300): d = 6, baker, n = 1000003, m = 32: 2.82 -> 0.55 ms; d = 8,
// Korobov 3, n = 4194301, m = 16: 20.4 -> 3.02 ms (2.98 without the peaked
// integrands' branch); per-shift values within 2e-16 of a 64-bit evaluation on both
// sides.
//
// What bounds it now: issue slots, 78 multiply-adds of four and 295 others a value
// at d = 6.  Tried: one row per CTA (d = 8: 4.47 ms), three CTAs per SM at 80
// registers (no gain), every slot of F without the mask (d = 8: 3.03 against
// 3.08 ms, but batches of sparse sectors 4.31 against 4.16 ms).
//
// Rows of two shifts are evaluated side by side (independent chains); a CTA
// takes one pair of shift rows, so few shifts on a small lattice still spread
// over the chip.
#pragma once

#include "rule_kernels.cuh"

namespace qmc {

constexpr int kFxShiftMin = 4;        // 2 su + sf of the largest U < 2^63 and F < 2^62 (leading zeros 1 and 2)
constexpr double kFxRange = 1000.0;   // largest (coefficient sum) / (constant term) of U and of F
constexpr double kFxPeaked = 64.0;    // the same, above which the Korobov weight is normalised

// a b + c, one multiply-add (spelled out: as a plain expression the compiler
// splits sums of such products into products and adds)
__host__ __device__ __forceinline__ uint64_t fx_mad(uint32_t a, uint32_t b, uint64_t c) {
#ifdef __CUDA_ARCH__
  uint64_t r;
  asm("mad.wide.u32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
  return r;
#else
  return (uint64_t)a * b + c;
#endif
}

// a b / 2^64 + c, the low words' product and the fractions of the cross products
// dropped (1.25 units on average, which k = 1.25 2^32 puts back)
__host__ __device__ __forceinline__ uint64_t fx_mulhi_add(uint64_t a, uint64_t b, uint64_t c, uint64_t k = 0) {
  const uint32_t al = (uint32_t)a, ah = (uint32_t)(a >> 32), bl = (uint32_t)b, bh = (uint32_t)(b >> 32);
  const uint64_t t1 = k ? fx_mad(al, bh, k) : (uint64_t)al * bh;
  const uint64_t t2 = (uint64_t)ah * bl;
  return fx_mad(ah, bh, c) + (t1 >> 32) + (t2 >> 32);
}

// the same for a, b < 2^63 with a + b < 2^64: the cross products' sum fits 64 bits
__host__ __device__ __forceinline__ uint64_t fx_mulhi63_add(uint64_t a, uint64_t b, uint64_t c) {
  const uint32_t al = (uint32_t)a, ah = (uint32_t)(a >> 32), bl = (uint32_t)b, bh = (uint32_t)(b >> 32);
  const uint64_t t = fx_mad(ah, bl, (uint64_t)al * bh);
  return fx_mad(ah, bh, c) + (t >> 32);
}

// a^2 / 2^64
__host__ __device__ __forceinline__ uint64_t fx_sqr(uint64_t a) {
  const uint32_t al = (uint32_t)a, ah = (uint32_t)(a >> 32);
  return (uint64_t)ah * ah + (((uint64_t)al * ah) >> 31);
}

__host__ __device__ __forceinline__ int fx_clz(uint64_t a) {  // leading zeros, a >= 2^32
#ifdef __CUDA_ARCH__
  return __clz((int)(uint32_t)(a >> 32));
#else
  return __builtin_clz((uint32_t)(a >> 32));
#endif
}

__host__ __device__ __forceinline__ int fx_clz64(uint64_t a) {  // leading zeros, 0 for a = 0
#ifdef __CUDA_ARCH__
  return __clzll((long long)a) & 63;
#else
  return a ? __builtin_clzll(a) : 0;
#endif
}

// 2^120 / y for y in [2^61, 2^64): a float reciprocal of the high word (error
// eps below 2^-22), then one third-order step r (1 + eps + eps^2) with eps to
// 2^-60 from the exact product.
__host__ __device__ __forceinline__ uint64_t fx_recip(uint64_t y) {
  const uint32_t yl = (uint32_t)y, yh = (uint32_t)(y >> 32);
#ifdef __CUDA_ARCH__
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(__uint2float_rn(yh)));
  const uint32_t r0 = __float2uint_rn(r * 0x1p60f);  // 2^92 / y within 2^-22
#else
  const uint32_t r0 = (uint32_t)(1.0f / (float)yh * 0x1p60f);
#endif
  const uint64_t p0 = (uint64_t)yl * r0;
  const uint64_t p1 = (uint64_t)yh * r0 + (p0 >> 32);            // y r0 / 2^32 = 2^60 (1 - eps)
  const int64_t e = (int64_t)((1ull << 60) - p1);                // eps 2^60
  const int32_t es = (int32_t)(e >> 8);                          // eps 2^52
  const uint32_t e2 = (uint32_t)((uint64_t)((int64_t)es * es) >> 32) >> 12;  // eps^2 2^60
  const uint64_t dl = (uint64_t)e + (1ull << 40) + e2;           // (eps + eps^2 + 2^-20) 2^60 >= 0
  const uint64_t q0 = (uint64_t)(uint32_t)dl * r0 + 0x80000000ull;
  const uint64_t q1 = (uint64_t)(uint32_t)(dl >> 32) * r0 + (q0 >> 32);
  return (uint64_t)r0 * ((1u << 28) - (1u << 8)) + q1;
}

// a with all bits flipped where the 32-bit mask m is all ones
__host__ __device__ __forceinline__ uint64_t fx_flip(uint64_t a, uint32_t m) {
  return ((uint64_t)((uint32_t)(a >> 32) ^ m) << 32) | ((uint32_t)a ^ m);
}

// Transformed coordinate (Q63) of the 64-bit fraction X; under Korobov 3 the
// factor 4x(1-x) (Q64) goes to u.  With v = |2x - 1|, u = 1 - v^2, Eq. (5)'s
// polynomial for weight 3 is z = 1/2 +- v (16 + 8u + 6u^2 + 5u^3) / 32, all
// terms positive.
template <int TR>
__host__ __device__ __forceinline__ uint64_t fx_coord(uint64_t X, uint64_t& u) {
  if constexpr (TR == TR_NONE) {
    return X >> 1;
  } else if constexpr (TR == TR_BAKER) {
    return fx_flip(X, (uint32_t)((int64_t)X >> 63));  // min(X, 2^64 - 1 - X) = 2^63 z
  } else {
    const uint32_t low = ~(uint32_t)((int64_t)X >> 63);  // all ones on the lower half
    const uint64_t v = fx_flip(X + X, low);
    u = ~fx_sqr(v);
    // (16 + 6u^2) / 64 + u (8 + 5u^2) / 64: one square and one product; the
    // constant is two units low, so that u's last bit cannot push z past 0 or 1
    const uint64_t q = fx_sqr(u) >> 6;
    const uint64_t h = fx_mulhi_add(u, q * 4 + q + 0x2000000000000000ull,
                                    (q * 2 + q) * 2 + (0x4000000000000000ull - 2));
    const uint64_t zv = fx_mulhi_add(v, h, 0);
    return fx_flip(zv, low) + 0x4000000000000000ull;
  }
}

// The Korobov coordinate for users that convert it to double: fx_coord's truncations
// leave z 6.5 units too large on average near 0, where a unit counts most (7.5 too
// small near 1).  The sectors take that off their constants.
__host__ __device__ __forceinline__ uint64_t fx_coord_centred(uint64_t X, uint64_t& u) {
  const uint64_t z = fx_coord<TR_KOROBOV>(X, u);
  return z > 6 ? z - 6 : 0;
}

// sum_j c_j z_j / 2^64 for constants c_j = (high word, low word / 16) with
// sum_j c_j < 2^64 and z_j < 2^63: with 28-bit low words the cross products of
// up to eight terms share one 64-bit sum, so a term is three multiply-adds and
// nothing else.
struct FxDot {
  uint64_t hi, t;
  __host__ __device__ __forceinline__ void add(uint64_t z, uint32_t ch, uint32_t cl) {
    const uint32_t zl = (uint32_t)z >> 4, zh = (uint32_t)(z >> 32);
    hi = fx_mad(zh, ch, hi);
    t = fx_mad(zl, ch, t);
    t = fx_mad(zh, cl, t);
  }
  __host__ __device__ __forceinline__ uint64_t value() const { return hi + (t >> 28); }
};

// NS weighted values at one point: v[s] 2^t[s] in units of value_scale.  TERM
// (single terms listed by the caller): the weight keeps its leading zeros
// apart, factor by factor, so a term of any size comes back to full relative
// precision.  In the rule's sums it does so for peaked integrands, after each half
// of the factors; for the others the weight's 2^-64 absolute steps are below the
// rounding of the sum's final conversion.  t[s] is negative only where the weight
// is normalised.
template <int D, int TR, int NS, bool TERM = false>
__host__ __device__ __forceinline__ void fx_values(const FxParams& P, const uint64_t* base, const uint64_t (*shift)[D],
                                                   uint64_t* v, int* t) {
  // two products of factors, so that four at most multiply unnormalised
  constexpr int H = D > 4 ? D / 2 : D;
  uint64_t z[NS][D], W[NS], W2[NS];
  int ew[NS];
#pragma unroll
  for (int i = 0; i < D; ++i)
#pragma unroll
    for (int s = 0; s < NS; ++s) {
      uint64_t u = 0;
      z[s][i] = fx_coord<TR>(base[i] + shift[s][i], u);
      if constexpr (TR == TR_KOROBOV) {
        if constexpr (TERM) {
          const int su = fx_clz64(u);
          u <<= su;
          W[s] = i == 0 ? u : fx_mulhi_add(W[s], u, 0);
          const int sw = fx_clz64(W[s]);
          W[s] <<= sw;
          ew[s] = (i == 0 ? 0 : ew[s]) + su + sw;
        } else if (i < H) {
          W[s] = i == 0 ? u : fx_mulhi_add(W[s], u, 0);
        } else {
          W2[s] = i == H ? u : fx_mulhi_add(W2[s], u, 0);
        }
      }
    }
  if constexpr (TR == TR_KOROBOV && !TERM) {
#pragma unroll
    for (int s = 0; s < NS; ++s) ew[s] = 0;
    const auto normalise = [&](uint64_t* w) {
#pragma unroll
      for (int s = 0; s < NS; ++s) {
        const int sw = fx_clz64(w[s]);
        w[s] <<= sw;
        ew[s] += sw;
      }
    };
    if (P.peaked) {
      normalise(W);
      if constexpr (H < D) normalise(W2);
    }
    if constexpr (H < D)
#pragma unroll
      for (int s = 0; s < NS; ++s) W[s] = fx_mulhi_add(W[s], W2[s], 0);
  }
  uint64_t U[NS], F[NS];
  FxDot dot[NS];
#pragma unroll
  for (int s = 0; s < NS; ++s) dot[s] = FxDot{P.u0, 0};
#pragma unroll
  for (int i = 0; i < D; ++i)
#pragma unroll
    for (int s = 0; s < NS; ++s) dot[s].add(z[s][i], P.uh[i], P.ul[i]);
#pragma unroll
  for (int s = 0; s < NS; ++s) {
    U[s] = dot[s].value();
    F[s] = P.f0;
  }
  // F row by row; a bit per slot (the row itself first) tells which terms
  // exist: a test and a branch (2 slots a pair of shifts) against 24
  int off = 0;
#pragma unroll
  for (int i = 0; i < D; ++i) {
    const uint32_t row = P.fmask[i];
    if (row) {
#pragma unroll
      for (int s = 0; s < NS; ++s) dot[s] = FxDot{P.fl[i], 0};
#pragma unroll
      for (int j = i; j < D; ++j)
        if (row & (2u << (j - i)))
#pragma unroll
          for (int s = 0; s < NS; ++s) dot[s].add(z[s][j], P.fh[off + j - i], P.fq[off + j - i]);
#pragma unroll
      for (int s = 0; s < NS; ++s) F[s] = fx_mulhi63_add(z[s][i], dot[s].value(), F[s]);
    }
    off += D - i;
  }
#pragma unroll
  for (int s = 0; s < NS; ++s) {
    const int su = fx_clz(U[s]), sf = fx_clz(F[s]);
    uint64_t r = fx_recip(fx_mulhi_add(fx_sqr(U[s] << su), F[s] << sf, 0));
    // the reciprocal is below 2^59: 4 more bits before the weight (0.2% on average at d = 8) takes them away
    if constexpr (TR == TR_KOROBOV) r = fx_mulhi_add(r << 4, fx_mulhi_add(fx_sqr(W[s]), W[s], 0), 0, 0x140000000ull);
    v[s] = r;
    t[s] = 2 * su + sf - kFxShiftMin - (TR == TR_KOROBOV ? 3 * ew[s] : 0);
  }
}

// 128-bit sum
struct FxSum {
  uint64_t lo, hi;
  __device__ __forceinline__ void add(uint64_t l, uint64_t h) {
    asm("add.cc.u64 %0, %0, %2;\n\taddc.u64 %1, %1, %3;" : "+l"(lo), "+l"(hi) : "l"(l), "l"(h));
  }
};

// idx / n to 96 bits (low 32 bits of the fraction in lo, the upper 64 returned)
__device__ __forceinline__ uint64_t fx_frac96(uint32_t idx, const Recip& rc, uint32_t& lo) {
  const uint64_t l = (uint64_t)idx * rc.rlo;
  lo = (uint32_t)(l >> 32);
  return frac64(idx, rc);
}

// A thread's successive points, kThreads apart: the fractions advance by a 96-bit
// add modulo 1.
template <int D>
struct FxWalk96 {
  uint64_t base[D];
  uint32_t lo[D];
  __device__ __forceinline__ void start(const FxBase& P, uint64_t j) {
#pragma unroll
    for (int i = 0; i < D; ++i) base[i] = fx_frac96(lattice_index(j, P.g[i], P.n), P.rc, lo[i]);
  }
  __device__ __forceinline__ void step(const FxBase& P) {
#pragma unroll
    for (int i = 0; i < D; ++i) {
      uint32_t mid = (uint32_t)base[i], top = (uint32_t)(base[i] >> 32);
      asm("add.cc.u32 %0, %0, %3;\n\taddc.cc.u32 %1, %1, %4;\n\taddc.u32 %2, %2, %5;"
          : "+r"(lo[i]), "+r"(mid), "+r"(top)
          : "r"(P.step[i][0]), "r"(P.step[i][1]), "r"(P.step[i][2]));
      base[i] = ((uint64_t)top << 32) | mid;
    }
  }
};

template <int D, int TR>
__global__ void __launch_bounds__(kThreads)
    sector_fx_kernel(const __grid_constant__ FxParams P, double* __restrict__ partial,
                     unsigned long long* __restrict__ counters, const SampleIO sio) {
  constexpr int NS = kFxRows;
  if (sio.count > 0) {
    int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= sio.count) return;
    const uint64_t j = sio.j[s];
    const int k = sio.k[s];
    uint64_t base[D], sh[1][D];
#pragma unroll
    for (int i = 0; i < D; ++i) {
      const uint32_t idx = lattice_index(j, P.g[i], P.n);
      base[i] = frac64(idx, P.rc);
      sh[0][i] = P.shift[k][i];
      if (sio.idx) sio.idx[(size_t)s * D + i] = idx;
      if (sio.coord) sio.coord[(size_t)s * D + i] = coord_used<double>(base[i] + P.shift[k][i]);
    }
    uint64_t v;
    int t;
    fx_values<D, TR, 1, true>(P, base, sh, &v, &t);
    sio.values[2 * (size_t)s] = ldexp(__ull2double_rn(v), t) * P.value_scale;
    sio.values[2 * (size_t)s + 1] = 0.0;
    return;
  }
  const int r0 = blockIdx.y * NS;
  uint64_t sh[NS][D];
#pragma unroll
  for (int s = 0; s < NS; ++s)
#pragma unroll
    for (int i = 0; i < D; ++i) sh[s][i] = P.shift[r0 + s][i];
  FxSum acc[NS];
#pragma unroll
  for (int s = 0; s < NS; ++s) acc[s].lo = acc[s].hi = 0;
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
      uint64_t v[NS];
      int t[NS];
      fx_values<D, TR, NS>(P, walk.base, sh, v, t);
#pragma unroll
      for (int q = 0; q < NS; ++q) {
        if (TR == TR_KOROBOV && P.peaked && t[q] < 0) acc[q].add(t[q] > -64 ? v[q] >> -t[q] : 0, 0);
        else acc[q].add(v[q] << t[q], __funnelshift_l((uint32_t)(v[q] >> 32), 0u, t[q]));
      }
      walk.step(P);
    }
  }
  // exact integer sums over the CTA, one conversion per slot
  __shared__ uint64_t red[kThreads / 32][NS][2];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
  for (int s = 0; s < NS; ++s) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const uint64_t l = __shfl_down_sync(0xffffffffu, acc[s].lo, o), h = __shfl_down_sync(0xffffffffu, acc[s].hi, o);
      acc[s].add(l, h);
    }
    if (lane == 0) {
      red[warp][s][0] = acc[s].lo;
      red[warp][s][1] = acc[s].hi;
    }
  }
  __syncthreads();
  if (threadIdx.x < NS && r0 + (int)threadIdx.x < P.m_launch) {
    FxSum tot{0, 0};
#pragma unroll
    for (int w = 0; w < kThreads / 32; ++w) tot.add(red[w][threadIdx.x][0], red[w][threadIdx.x][1]);
    const size_t slot = ((size_t)(P.k_base + r0 + threadIdx.x) * P.nblk + blockIdx.x) * 2;
    partial[slot] = fma(__ull2double_rn(tot.hi), 0x1p64, __ull2double_rn(tot.lo));
    partial[slot + 1] = 0.0;
  }
}

}  // namespace qmc
