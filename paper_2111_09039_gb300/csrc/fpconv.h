// Device helpers for the element-wise kernels on n x k blocks.
//
// FP64 instructions issue at a 64th of the FP32 rate on this GPU (a warp's takes 64
// clocks of its sub-partition alone, 76 where all four issue FMAs back to back, 69 in
// S X), and the FP64 <-> FP32 conversion instructions are not free either, so conversions
// on the hot blocks are done on the bit patterns with integer operations, for
// every input: a conversion instruction on a rare path is predicated by the
// compiler and takes its 64 to 76 clocks of the FP64 pipe per warp whether any lane
// needs it or not (250,000 x 720 Rayleigh quotients with three conversions per
// entry: 1.00 ms, 0.73 ms without, in the sums' form of that time; residual sums of
// 250,000 x 500 1.18 and 0.45 ms; FP32 residuals with diagonal M 1.05 and 0.69 ms).
#pragma once

#include <cuda_runtime.h>

namespace hsim {
namespace k {

// FP64 -> FP32 with the significand truncated; results below the FP32 normal
// range are rounded to nearest (ties to even), those above it infinite
__device__ __forceinline__ float d2f_trunc(double v) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(v);
    const unsigned hi = (unsigned)(b >> 32), sign = hi & 0x80000000u;
    const int e = (int)((hi >> 20) & 0x7ff);
    if (e < 1023 - 126 || e > 1023 + 127) {
        const unsigned long long m = b & 0xfffffffffffffull;
        if (e > 1023 + 127) return __uint_as_float(e == 0x7ff && m ? 0x7fffffffu : sign | 0x7f800000u);
        const int s = 1023 - 126 - e + 29;  // 30 and more
        if (e == 0 || s > 54) return __uint_as_float(sign);
        const unsigned long long M = m | 0x10000000000000ull, q = M >> s, rest = M & ((1ull << s) - 1), half = 1ull << (s - 1);
        return __uint_as_float(sign | ((unsigned)q + (rest > half || (rest == half && (q & 1)) ? 1u : 0u)));
    }
    return __uint_as_float(sign | ((unsigned)(e - 896) << 23) | (unsigned)((b >> 29) & 0x7fffffu));
}

// exact FP32 -> FP64 of finite values
__device__ __forceinline__ double f2d_bits(float x) {
    const unsigned u = __float_as_uint(x);
    unsigned e = (u >> 23) & 0xffu, m = u & 0x7fffffu;
    if (e == 0u) {
        if (m == 0u) return __hiloint2double((int)(u & 0x80000000u), 0);
        const int up = __clz(m) - 8;  // subnormal: leading bit to position 23
        m = (m << up) & 0x7fffffu;
        e = (unsigned)(1 - up);       // 0 .. -22, of 896 + e
    }
    return __hiloint2double((int)((u & 0x80000000u) | ((e + 896u) << 20) | (m >> 3)), (int)(m << 29));
}

// x 2^e by adding e to the exponent field; subnormals and results outside the
// normal range (rounded to nearest, ties to even) on the significand
__device__ __forceinline__ double scale2(double x, int e) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    int ex = (int)((b >> 52) & 0x7ff);
    if (ex == 0 || ex + e <= 0 || ex + e >= 2047) {
        const unsigned long long sign = b & 0x8000000000000000ull;
        unsigned long long m = b & 0xfffffffffffffull;
        if (ex == 0x7ff || (ex == 0 && m == 0)) return x;
        if (ex == 0) {
            const int up = __clzll((long long)m) - 11;
            m <<= up;
            ex = 1 - up;
        }
        m |= 0x10000000000000ull;
        const int E = ex + e;
        if (E >= 2047) return __longlong_as_double((long long)(sign | 0x7ff0000000000000ull));
        if (E > 0) return __longlong_as_double((long long)(sign | (m & 0xfffffffffffffull) | ((unsigned long long)E << 52)));
        const int s = 1 - E;
        if (s > 53) return __longlong_as_double((long long)sign);
        const unsigned long long q = m >> s, rest = m & ((1ull << s) - 1), half = 1ull << (s - 1);
        return __longlong_as_double((long long)(sign | (q + (rest > half || (rest == half && (q & 1)) ? 1u : 0u))));
    }
    return __longlong_as_double((long long)(b + ((unsigned long long)(long long)e << 52)));
}

}  // namespace k
}  // namespace hsim

// rows strided over blockIdx.y, columns over blockIdx.x * blockDim.x +
// threadIdx.x (no index division); launch with grid_rc
#define HSIM_FOR_RC(i, rows, j, cols)                                                   \
    for (int i = blockIdx.y; i < (rows); i += gridDim.y)                                \
        for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < (cols); j += gridDim.x * blockDim.x)

// the same with the loads of four rows in flight (the grid covers the columns)
#define HSIM_ROWS_OF_COLUMN(i, rows, j, cols)                                           \
    const int j = blockIdx.x * blockDim.x + threadIdx.x;                                \
    if (j >= (cols)) return;                                                            \
    _Pragma("unroll 4") for (int i = blockIdx.y; i < (rows); i += gridDim.y)

// at most 2048 row strides: each block walks many rows (launching one block
// per row of a 10^6-row block spends the time in block scheduling)
inline dim3 grid_rc(int rows, int cols, int threads = 256) {
    const int cx = (cols + threads - 1) / threads;
    const int ry = rows < 2048 ? (rows > 0 ? rows : 1) : 2048;
    return dim3((unsigned)(cx > 0 ? cx : 1), (unsigned)ry);
}
