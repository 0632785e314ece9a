// Final deterministic pass of the rule on the GPU: per-shift CTA slots ->
// Q^(k) (Eq. 2), Qbar and the two-pass sigma^2 (Eq. 3).
#include "kernel_table.h"
#include "device_common.cuh"

namespace qmc {

// Latency bounds this pass: a few thousand slots, then chains of dependent FP64
// operations.  So every (shift, part) has its own warp up to 32 of them,
// a lane's loads are issued eight at a time before they are added (in the fixed
// order of the slots), and the two parts of Eq. (3) run in two warps.
// With 8 warps, one load at a time and one scaling per warp it took 11.3 us at m =
// 10 (now 8.7), and 47 us (now 10.6) for 16 shared-lattice sectors and their sum,
// whose slots the sweeps now write.

// s plus the slots lane, lane + 32, ... of one shift's part, in that order
__device__ __forceinline__ double add_slots(double s, const double* p, int nblk, int lane) {
  for (int b = lane; b < nblk; b += 8 * 32) {
    double v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) v[u] = b + 32 * u < nblk ? p[2 * (size_t)(b + 32 * u)] : 0.0;
#pragma unroll
    for (int u = 0; u < 8; ++u)
      if (b + 32 * u < nblk) s += v[u];
  }
  return s;
}

// One CTA per problem (per group of a problem: the epsilon orders of one
// pass have their slots, counters and results one after another).  Warp w
// adds the CTA slots of (shift, part) tasks w, w + 32, ... in a fixed order;
// warps 0 and 1 then form Qbar and the two-pass sigma^2 of the two parts.
__device__ void finalize_one(FinalizeArgs A, int grp, double* q /* shared [m][2] */) {
  A.partial += (size_t)grp * A.m * A.nblk * 2;
  A.counters += 2 * grp;
  A.result += grp;
  if (A.per_shift) A.per_shift += (size_t)grp * A.m * 2;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int parts = A.is_complex ? 2 : 1;
  const int tasks = A.m * parts;
  for (int t = warp; t < tasks; t += kFinThreads / 32) {
    const int k = t / parts, part = t % parts;
    const double s = warp_sum_d(add_slots(0.0, A.partial + (size_t)k * A.nblk * 2 + part, A.nblk, lane));
    if (lane == 0) q[2 * k + part] = s;
  }
  __syncthreads();
  for (int t = threadIdx.x; t < 2 * A.m; t += kFinThreads) {
    const int part = t & 1;
    q[t] = part < parts ? (q[t] * A.value_scale) / A.dn + A.offset[part] : A.offset[1];
  }
  __syncthreads();
  if (warp < 2) {
    const int part = warp;
    double s = 0.0;
    for (int k = lane; k < A.m; k += 32) s += q[2 * k + part];
    s = warp_sum_d(s);
    const double mean = __shfl_sync(0xffffffffu, s, 0) / (double)A.m;
    double v = 0.0;
    for (int k = lane; k < A.m; k += 32) {
      double dlt = q[2 * k + part] - mean;
      v = fma(dlt, dlt, v);
    }
    v = warp_sum_d(v);
    if (lane == 0) {
      const double var = v / ((double)A.m * (double)(A.m - 1));
      A.result->mean[part] = mean;
      A.result->var[part] = var;
      A.result->err[part] = sqrt(var);
    }
  } else {
    if (A.per_shift)
      for (int t = threadIdx.x - 64; t < 2 * A.m; t += kFinThreads - 64) A.per_shift[t] = q[t];
    if (threadIdx.x == 64) {
      const unsigned long long nf = A.counters[0], dv = A.counters[1];
      A.result->nonfinite = nf;
      A.result->deform_violations = dv;
      A.result->status = nf ? QMC_ENONFINITE : (dv ? QMC_EDEFORM : QMC_OK);
      A.result->reserved = 0;
      A.counters[0] = 0;
      A.counters[1] = 0;
    }
  }
}

__global__ void __launch_bounds__(kFinThreads) finalize_kernel(const FinalizeArgs A) {
  extern __shared__ double q[];
  finalize_one(A, blockIdx.x, q);
}

// Batched final pass: CTA b finalises problem b.
__global__ void __launch_bounds__(kFinThreads) finalize_batch_kernel(const FinalizeArgs* __restrict__ args) {
  extern __shared__ double q[];
  finalize_one(args[blockIdx.x], 0, q);
}

const void* finalize_ptr() { return (const void*)&finalize_kernel; }
const void* finalize_batch_ptr() { return (const void*)&finalize_batch_kernel; }

}  // namespace qmc
