// The tensor-core class on tcgen05, first pass of four-step plans (UmmaBody mode
// 1, or 3: tc_columns_fused): 2^7 .. 2^10 points, complex64 and complex32.
#include "umma_kernel.cuh"

namespace gbfft {

const void* resolve_umma_cols1(int logL, int prec, int io16) {
#define GB_UMMA(LG)                                                        \
  if (logL == LG) {                                                        \
    if (io16) return (const void*)stockham_umma<LG, TC_FP16, true, 1>;     \
    if (prec == TC_FP16) return (const void*)stockham_umma<LG, TC_FP16, false, 3>; \
    if (prec == TC_BF16) return (const void*)stockham_umma<LG, TC_BF16, false, 3>; \
    return (const void*)stockham_umma<LG, TC_BF16X3, false, 1>;            \
  }
  GB_UMMA(7) GB_UMMA(8) GB_UMMA(9) GB_UMMA(10)
#undef GB_UMMA
  return nullptr;
}

}  // namespace gbfft
