// complex128 resident 1D step kernels, N = 64 .. 2048
#include "soft1d_c128_list.h"
#include "soft1d_inst.cuh"
namespace soft {
Launch1D soft1d_c128_a(int logn, int loge, int logrm) {
    SOFT1D_CASE(double, 6, 1, 1)
    SOFT1D_CASE(double, 7, 2, 2)
#define CASE(LN, LE, LRM) SOFT1D_CASE(double, LN, LE, LRM)
    SOFT1D_C128_256_TO_2048(CASE)
#undef CASE
    return nullptr;
}
}  // namespace soft
