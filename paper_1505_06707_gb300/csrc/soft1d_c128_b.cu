// complex128 resident 1D step kernels, N = 4096 .. 16384
#include "soft1d_c128_list.h"
#include "soft1d_inst.cuh"
namespace soft {
Launch1D soft1d_c128_b(int logn, int loge, int logrm) {
#define CASE(LN, LE, LRM) SOFT1D_CASE(double, LN, LE, LRM)
    SOFT1D_C128_4096_TO_8192(CASE)
#undef CASE
    SOFT1D_CASE(double, 14, 5, 4)
    return nullptr;
}
}  // namespace soft
