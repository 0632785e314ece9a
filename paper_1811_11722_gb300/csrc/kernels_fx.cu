// Instantiations of the fixed-point FP64 sector kernel for one d, compiled
// once per d with -DQMC_D=1..8.
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

}  // namespace qmc
