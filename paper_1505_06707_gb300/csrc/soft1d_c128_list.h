// The built (LOGN, LOGE, LOGRM) variants of the complex128 1D step from N = 256
// to N = 8192: the step kernels (soft1d_c128_*.cu) and the surface-sampled step
// (soft1d_surf.cu) are built from one list, because tuning may give a single
// plan any of them.
#pragma once

#define SOFT1D_C128_256_TO_2048(X) \
    X(8, 2, 2) X(8, 3, 3) X(9, 2, 2) X(9, 3, 3) X(10, 2, 2) X(10, 3, 3) X(10, 4, 4) X(11, 3, 3) X(11, 4, 4)
#define SOFT1D_C128_4096_TO_8192(X) X(12, 3, 3) X(12, 4, 4) X(13, 4, 4)
