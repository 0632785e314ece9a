// Instantiations of the fixed-point FP64 kernels (sector, deformed) for one d,
// compiled once per d with -DQMC_D=1..8.
#include "deformed_fx.cuh"
#include "fixed64.cuh"
#include "kernel_table.h"

#ifndef QMC_D
#error "QMC_D must be 1..8"
#endif

namespace qmc {

template <>
const void* sector_fx_ptr<QMC_D>(int tr) {
  if (tr == TR_NONE) return (const void*)&sector_fx_kernel<QMC_D, TR_NONE>;
  if (tr == TR_BAKER) return (const void*)&sector_fx_kernel<QMC_D, TR_BAKER>;
  if (tr == TR_KOROBOV) return (const void*)&sector_fx_kernel<QMC_D, TR_KOROBOV>;
  return nullptr;
}

template <>
const void* deformed_fx_ptr<QMC_D>() {
  if constexpr (QMC_D <= kDefFxMax) return (const void*)&deformed_fx_kernel<QMC_D>;
  else return nullptr;
}

}  // namespace qmc
