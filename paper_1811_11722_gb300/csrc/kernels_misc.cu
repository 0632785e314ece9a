// Separable and general rule kernels for one precision (compiled once per
// precision with -DQMC_REAL=float|double).
#include "kernel_table.h"
#include "rule_kernels.cuh"
#include "separable64.cuh"

#ifndef QMC_REAL
#error "QMC_REAL must be float or double"
#endif

namespace qmc {

#define QMC_SEP_FK(K, ...)                                             \
  do {                                                                 \
    if (fk == FK_CONST) return (const void*)&K<__VA_ARGS__, FK_CONST>;   \
    if (fk == FK_SEPEXP) return (const void*)&K<__VA_ARGS__, FK_SEPEXP>; \
    if (fk == FK_TRIG) return (const void*)&K<__VA_ARGS__, FK_TRIG>;     \
  } while (0)

// FP64: one shift row per CTA row (separable64.cuh); FP32: 8 shifts per thread.
template <>
const void* separable_ptr_t<QMC_REAL>(int tr, bool fixed, int fk) {
  if constexpr (sizeof(QMC_REAL) == 8) {
    if (tr == TR_NONE) QMC_SEP_FK(separable64_kernel, TR_NONE, false);
    if (tr == TR_BAKER) QMC_SEP_FK(separable64_kernel, TR_BAKER, false);
    if (tr == TR_KOROBOV && fixed) QMC_SEP_FK(separable64_kernel, TR_KOROBOV, true);
    if (tr == TR_KOROBOV) QMC_SEP_FK(separable64_kernel, TR_KOROBOV, false);
  } else {
    if (tr == TR_NONE) QMC_SEP_FK(separable_kernel, QMC_REAL, 8, TR_NONE);
    if (tr == TR_BAKER) QMC_SEP_FK(separable_kernel, QMC_REAL, 8, TR_BAKER);
    if (tr == TR_KOROBOV) QMC_SEP_FK(separable_kernel, QMC_REAL, 8, TR_KOROBOV);
  }
  return nullptr;
}

template <>
const void* general_ptr_t<QMC_REAL>() {
  return (const void*)&general_kernel<QMC_REAL, 8>;
}

template <>
const void* general_eps_ptr_t<QMC_REAL>() {
  return (const void*)&general_eps_kernel<QMC_REAL>;
}

}  // namespace qmc
