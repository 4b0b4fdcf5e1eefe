// Weight and bias gradients of the 3x3 convolutions on the tensor cores:
//   dW[o][c][tap] = sum_p g[p][o] in[p + tap][c],  db[o] = sum_p g[p][o],
// a contraction over pixels, M = output channels, N = (tap, input channel),
// K = pixels, by warp mma.sync m16n8k16 (BF16 operands, FP32 accumulators).
// Both operands lie in memory with the channels of a pixel contiguous, so
// their fragments are transposed ldmatrix loads of the rows as they are, and a
// tap only moves the pixel a load starts at.  (tcgen05 wants M of 64 or more
// in one core-matrix stride; 32 channels x 9 taps have two strides and would
// need an im2col copy, which costs more than the products.)
//
// FP32 operands (the network's input, the loss gradient) enter as three BF16
// terms that add up to them exactly (8 + 8 + 8 bits), so the products are
// those of the FP32 value.  The tensor cores' FP32 accumulation truncates, a
// bias that grows with the chain: 8 products deep it left 5.5e-8 of the gradient
// of exact operands (32 fields of 128^2), the scalar sums 2.3e-8.  So each
// product starts from zero, where the sum of 16 terms of 16 bits loses little,
// and is added, rounded to nearest, to the thread's sums in registers; the CTAs'
// sums are added in FP64.  2.3e-8, as the scalar sums, and less on small fields
// (3 x 128: 3.5e-8 against 9.1e-8); the additions cost less than the
// shared-memory sums that 8-product chains were added to (a gradient of 32
// fields of 128^2: 425 -> 411 us).
//
// The scalar form took 7.4 of the 7.7 ms of a gradient on 32 fields of 128^2:
// two shared-memory loads per multiply-add.  These kernels read each row
// once (cp.async, the next row in flight during the products).
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "conv.cuh"
#include "device_common.cuh"

namespace soft {

enum WgKind { WG_BF16_32 = 0, WG_SPLIT = 1 };     // 32 BF16 channels; 2 FP32 channels split in three

__device__ __forceinline__ void ldsm_x4_t(uint32_t (&r)[4], const void* p) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"((uint32_t)__cvta_generic_to_shared(p)));
}
__device__ __forceinline__ void ldsm_x2_t(uint32_t (&r)[2], const void* p) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0,%1}, [%2];"
                 : "=r"(r[0]), "=r"(r[1]) : "r"((uint32_t)__cvta_generic_to_shared(p)));
}
// (x, y) = sum of three BF16 pairs, exactly (to 2^-24 relative)
__device__ __forceinline__ void split3(float2 v, uint32_t* s) {
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const __nv_bfloat162 b = __floats2bfloat162_rn(v.x, v.y);
        s[k] = *reinterpret_cast<const uint32_t*>(&b);
        v.x -= __bfloat162float(b.x);
        v.y -= __bfloat162float(b.y);
    }
}

// d = a b, rounded toward zero by the tensor core, into fresh accumulators
__device__ __forceinline__ void mma_bf16_zero(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 "
        "{%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%10,%10,%10};\n"
        : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1), "f"(0.0f));
}

template <int AK, int BK>
struct WgCfg {
    static constexpr int MT = AK == WG_BF16_32 ? 2 : 1;      // m16 tiles: 32 outputs, or 2 x 3 terms
    static constexpr int NB = BK == WG_BF16_32 ? 4 : 1;      // n8 tiles per tap: 32 inputs, or 2 x 3 terms
    static constexpr int COUT = AK == WG_BF16_32 ? 32 : 2, CIN = BK == WG_BF16_32 ? 32 : 2;
    static constexpr int NW = COUT * CIN * 9, NP = NW + COUT;
    // bytes per pixel in shared memory: eight consecutive pixels of a
    // fragment load fall in different banks
    static constexpr int AP = AK == WG_BF16_32 ? 80 : 48, BP = BK == WG_BF16_32 ? 80 : 16;
    static constexpr int AROW = 128 * AP, BROW = 130 * BP;
    static constexpr int THREADS = 384;                      // warps: 3 tap rows x 4 pixel groups
    static constexpr int COLS = 9 * NB * 8 + 1;              // products, then the bias column
    static constexpr int RED = MT * 16 * COLS * 4;
    static constexpr int TILES = 2 * AROW + 4 * BROW;
    static_assert(RED <= TILES, "the final sums reuse the tiles' memory");
    static constexpr int SMEM = TILES;
    static constexpr int MAXROWS = 64;                       // rows of 128 pixels per CTA
};

// Rows r0 .. r0 + rows - 1 of the list (field, 128-pixel segment, y), y
// fastest; partial sums in parameter order at part[blockIdx.x * NP].
template <int AK, int BK>
__global__ void __launch_bounds__(384)
wgrad_tc_kernel(const void* __restrict__ in, const void* __restrict__ gout, int H, int W, int64_t nrows, int rows,
                float* __restrict__ part)
{
    using Q = WgCfg<AK, BK>;
    constexpr int MT = Q::MT, NB = Q::NB;
    extern __shared__ __align__(16) unsigned char sm[];
    unsigned char* ga = sm;                      // [2][128][AP]
    unsigned char* xb = sm + 2 * Q::AROW;        // [4][130][BP]
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int dy = warp >> 2, ks = warp & 3;
    const int64_t r0 = (int64_t)blockIdx.x * rows, r1 = r0 + rows < nrows ? r0 + rows : nrows;
    const int nseg = W / 128;

    auto load_b = [&](int slot, int64_t f, int x0, int y) {        // input row y (periodic), pixels x0-1 .. x0+128
        y = y < 0 ? y + H : (y >= H ? y - H : y);
        const int64_t base = (f * H + y) * W;
        unsigned char* dst = xb + slot * Q::BROW;
        if constexpr (BK == WG_BF16_32) {
            for (int i = tid; i < 130 * 4; i += Q::THREADS) {
                const int px = i >> 2, q = i & 3;
                int x = x0 + px - 1;
                x = x < 0 ? x + W : (x >= W ? x - W : x);
                cp_async<16>(dst + px * Q::BP + q * 16, reinterpret_cast<const unsigned char*>(in) + (base + x) * 64 + q * 16);
            }
        } else {
            for (int px = tid; px < 130; px += Q::THREADS) {
                int x = x0 + px - 1;
                x = x < 0 ? x + W : (x >= W ? x - W : x);
                uint32_t s[3];
                split3(reinterpret_cast<const float2*>(in)[base + x], s);
                *reinterpret_cast<uint4*>(dst + px * Q::BP) = make_uint4(s[0], s[1], s[2], 0u);
            }
        }
    };
    auto load_a = [&](int slot, int64_t f, int x0, int y) {
        const int64_t base = (f * H + y) * W + x0;
        unsigned char* dst = ga + slot * Q::AROW;
        if constexpr (AK == WG_BF16_32) {
            for (int i = tid; i < 128 * 4; i += Q::THREADS)
                cp_async<16>(dst + (i >> 2) * Q::AP + (i & 3) * 16,
                             reinterpret_cast<const unsigned char*>(gout) + (base + (i >> 2)) * 64 + (i & 3) * 16);
        } else {
            for (int px = tid; px < 128; px += Q::THREADS) {
                uint32_t s[3];
                split3(reinterpret_cast<const float2*>(gout)[base + px], s);
                uint4* d = reinterpret_cast<uint4*>(dst + px * Q::AP);
                d[0] = make_uint4(s[0], s[1], s[2], 0u);
                d[1] = make_uint4(0u, 0u, 0u, 0u);
            }
        }
    };

    // acc[m][d][n]: tap column d, input tile n; acc[m][3 NB ...]: the bias
    constexpr int TL = 3 * NB + 1;
    float acc[MT][TL][4];
#pragma unroll
    for (int m = 0; m < MT; ++m)
#pragma unroll
        for (int n = 0; n < TL; ++n)
#pragma unroll
            for (int k = 0; k < 4; ++k) acc[m][n][k] = 0.0f;
    auto product = [&](float (&s)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
        float t[4];
        mma_bf16_zero(t, a, b0, b1);
#pragma unroll
        for (int k = 0; k < 4; ++k) s[k] += t[k];
    };
    const int mi = lane >> 3, mr = lane & 7;      // matrix and row of this lane's ldmatrix address
    int sb = 0, sa = 0;                           // ring slots of input row y - 1 and of g
    bool primed = false;
    for (int64_t r = r0; r < r1; ++r) {
        const int y = (int)(r % H);
        const int64_t fs = r / H, f = fs / nseg;
        const int x0 = (int)(fs % nseg) * 128;
        if (!primed) {
            for (int k = 0; k < 3; ++k) load_b((sb + k) & 3, f, x0, y - 1 + k);
            load_a(sa, f, x0, y);
            cp_async_commit();
            cp_async_wait<0>();
            __syncthreads();
        }
        const bool next = r + 1 < r1 && y + 1 < H;
        if (next) {
            load_b((sb + 3) & 3, f, x0, y + 2);
            load_a(sa ^ 1, f, x0, y + 1);
            cp_async_commit();
        }
        const unsigned char* A = ga + sa * Q::AROW;
        const unsigned char* B = xb + ((sb + dy) & 3) * Q::BROW;
#pragma unroll
        for (int q = ks; q < 8; q += 4) {
            uint32_t a[MT][4];
#pragma unroll
            for (int m = 0; m < MT; ++m)
                ldsm_x4_t(a[m], A + (16 * q + (mi >> 1) * 8 + mr) * Q::AP + m * 32 + (mi & 1) * 16);
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                if constexpr (NB == 4) {
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        uint32_t b[4];
                        ldsm_x4_t(b, B + (16 * q + d + (mi & 1) * 8 + mr) * Q::BP + h * 32 + (mi >> 1) * 16);
#pragma unroll
                        for (int m = 0; m < MT; ++m) {
                            product(acc[m][4 * d + 2 * h], a[m], b[0], b[1]);
                            product(acc[m][4 * d + 2 * h + 1], a[m], b[2], b[3]);
                        }
                    }
                } else {
                    uint32_t b[2];
                    ldsm_x2_t(b, B + (16 * q + d + (mi & 1) * 8 + mr) * Q::BP);
#pragma unroll
                    for (int m = 0; m < MT; ++m) product(acc[m][d], a[m], b[0], b[1]);
                }
            }
            if (dy == 1) {                        // bias: times ones
#pragma unroll
                for (int m = 0; m < MT; ++m) product(acc[m][TL - 1], a[m], 0x3f803f80u, 0x3f803f80u);
            }
        }
        cp_async_wait<0>();
        __syncthreads();
        primed = next;
        if (next) { sb = (sb + 1) & 3; sa ^= 1; }
    }
    // sum over the four pixel groups in shared memory: red[m][tap][n]
    float* red = reinterpret_cast<float*>(sm);
    const int g = lane >> 2, t = lane & 3;
    for (int k = 0; k < 4; ++k) {
        if (ks == k) {
#pragma unroll
            for (int m = 0; m < MT; ++m)
#pragma unroll
                for (int n = 0; n < TL; ++n)
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const bool bias = n == TL - 1;
                        if (bias && (dy != 1 || t != 0 || (e & 1))) continue;
                        const int col = bias ? 9 * NB * 8 : (dy * 3 * NB + n) * 8 + 2 * t + (e & 1);
                        float* p = &red[(m * 16 + g + (e >> 1) * 8) * Q::COLS + col];
                        const float v = acc[m][n][e];
                        *p = k == 0 ? v : *p + v;
                    }
        }
        __syncthreads();
    }
    float* out = part + (int64_t)blockIdx.x * Q::NP;
    constexpr int SA = AK == WG_SPLIT ? 3 : 1, SB = BK == WG_SPLIT ? 3 : 1;
    for (int i = tid; i < Q::NP; i += Q::THREADS) {
        const bool bias = i >= Q::NW;
        const int tap = i % 9, c = (i / 9) % Q::CIN, o = bias ? i - Q::NW : i / (9 * Q::CIN);
        const int col = bias ? 9 * NB * 8 : tap * NB * 8 + c;
        float s = 0.0f;
#pragma unroll
        for (int u = SA - 1; u >= 0; --u)        // the smallest terms first
            for (int v = (bias ? 1 : SB) - 1; v >= 0; --v) s += red[(o + 2 * u) * Q::COLS + col + 2 * v];
        out[i] = s;
    }
}

// sum of the CTA partials in FP64 (fixed order: eight strided sums, then their
// sum) into the gradient vector; 32 parameters per CTA of 256
__global__ void __launch_bounds__(256)
wgrad_reduce_kernel(const float* __restrict__ part, int ncta, int np, int nw, float* __restrict__ gW,
                    float* __restrict__ gb) {
    __shared__ double red[8][32];
    const int k = threadIdx.x >> 5, id = blockIdx.x * 32 + (threadIdx.x & 31);
    double s = 0;
    if (id < np)
        for (int c = k; c < ncta; c += 8) s += (double)part[(int64_t)c * np + id];
    red[k][threadIdx.x & 31] = s;
    __syncthreads();
    if (k == 0 && id < np) {
        for (int j = 1; j < 8; ++j) s += red[j][threadIdx.x];
        if (id < nw) gW[id] = (float)s;
        else gb[id - nw] = (float)s;
    }
}

}  // namespace soft
