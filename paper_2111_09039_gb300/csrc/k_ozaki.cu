// FP64-accurate dense products on BF16 tensor cores (error-free splitting).
//
// The Gram products S_bar = Psi^T S Psi, M_bar = Psi^T M Psi and the basis
// update Phi = Psi Phi_bar of Alg. 1 are the dominant dense work of the
// subspace iteration; in FP64 they run at the GB300's 1.2 TFLOP/s FP64 rate.
// Here each FP64 operand is split, against one power of two per row (or per
// column), into SL integer digits of at most 8 bits (SL = 7, 6, or 5 where 39
// bits suffice),
//     x = 2^(e-7) * sum_s d_s 2^(-8 s),   |d_0| <= 128, |d_s| <= 128,
// which BF16 represents exactly.  The tensor cores compute sum_r d_s(x_ir)
// d_t(y_jr) exactly, grouped by D = s + t (pairs with D >= ND are dropped, ND =
// SL for five and six digits, 8 for seven), and the groups are added into FP32
// expansions.  The result equals the FP64 product up to the truncation of the
// operands, about 2^-(8 SL - 1) of max|x_i.| max|y_j.| per term (2^-47 with six
// digits, 2^-55 with seven, the form that stands in for FP64 arithmetic).
//
// Kernel shape: C (FP64, M x N) (+)= X Y^T with X (M x K) and Y (N x K) both
// K-contiguous digit slices, on the tcgen05 tensor cores (TMA-fed shared
// memory, TMEM accumulators; k_ozaki_tc below).
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>

#include "common.h"
#include "fpconv.h"
#include "kernels.h"

namespace hsim {
namespace k {

namespace {

constexpr int kNoExp = -5000;     // exponent of a row or column of zeros
constexpr int kNonFinite = 1025;  // of an infinity or NaN
constexpr int kBadExp = 1 << 20;  // the same in a block whose rows or columns are scaled

inline unsigned cdiv(int64_t a, int64_t b) { return (unsigned)((a + b - 1) / b); }

// Exponents and digits are taken from the bits of the FP64 values with integer
// arithmetic only (the FP64 pipe of this part is a 64th of the FP32 pipe).
//
// smallest e with |x| < 2^e for a nonzero x: biased exponent - 1022 (subnormals
// by their leading bit); kNoExp for zero
__device__ __forceinline__ int exp_bits(double a) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(a) & 0x7FFFFFFFFFFFFFFFULL;
    const int e = (int)(b >> 52);
    if (e != 0) return e - 1022;
    return b == 0 ? kNoExp : -1010 - __clzll((long long)b);
}

// |x| 2^-e < 1 truncated to 24 bits (0 for subnormals and below 2^-126)
__device__ __forceinline__ float scaled_abs(double x, int e) {
    const unsigned h = (unsigned)__double2hiint(x) & 0x7FFFFFFFu, l = (unsigned)__double2loint(x);
    const int E = (int)(h >> 20), q = E - 1023 - e + 127;
    return E != 0 && q >= 1 && q < 127 ? __uint_as_float(((unsigned)q << 23) | ((h & 0xFFFFFu) << 3) | (l >> 29)) : 0.f;
}

// Limits of a row (column) in the check of an FP64 product's entries (digits_fail):
// infinite where it holds infinities or NaN, minus infinity where it is zero
__device__ __forceinline__ bool bad_exp(int e) { return e == kNonFinite || e >= kBadExp; }
__device__ __forceinline__ float entry_limit(int e, float sum) {
    return bad_exp(e) ? __int_as_float(0x7F800000) : e == kNoExp ? __int_as_float((int)0xFF800000) : sum;
}

// per-row exponents of a row-major R x C FP64 block: one warp per row; with
// cexp, of the block whose column c is scaled by 2^-cexp[c]; limits: entry_limit of
// the row's sum of |x| in units of 2^ex.  The upper words decide; subnormals count as
// 2^-1022 unless the row holds nothing else (and is not scaled).
__global__ void k_row_exps(int R, int C, const double *__restrict__ X, int ldx, const int *__restrict__ cexp,
                           int *__restrict__ ex, float *__restrict__ limits) {
    int row = blockIdx.x * (blockDim.x / 32) + threadIdx.x / 32;
    int lane = threadIdx.x & 31;
    if (row >= R) return;
    const double *x = X + (size_t)row * ldx;
    int m = kNoExp;
#pragma unroll 4
    for (int j = lane; j < C; j += 32) {
        const double v = x[j];
        const int h = __double2hiint(v) & 0x7FFFFFFF, c = cexp ? cexp[j] : 0;
        const int e = (h >> 20) - 1022 - c;
        m = max(m, (h | __double2loint(v)) == 0 ? kNoExp : cexp && h >= 0x7FF00000 ? kBadExp : e);
    }
    m = __reduce_max_sync(0xffffffffu, m);
    if (m == -1022 && !cexp) {
        m = kNoExp;
        for (int j = lane; j < C; j += 32) m = max(m, exp_bits(x[j]));
        m = __reduce_max_sync(0xffffffffu, m);
    }
    if (lane == 0) ex[row] = m;
    if (!limits) return;
    float s = 0.f;
#pragma unroll 4
    for (int j = lane; j < C; j += 32) s += scaled_abs(x[j], m + (cexp ? cexp[j] : 0));
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) limits[row] = entry_limit(m, s);
}

// h (upper word of |x|) added to a sum of magnitudes in units of 2^(ref - 1023),
// ref the biased exponent of the first normal value met (0: none yet); infinite
// where a later value is 2^127 times that
__device__ __forceinline__ void add_abs(unsigned h, int &ref, float &sum) {
    const int E = (int)(h >> 20);
    ref = ref != 0 ? ref : E;
    const int q = E - ref + 127;
    const float f = __uint_as_float((h << 3) + ((unsigned)(127 - ref) << 23));
    sum += q > 254 ? __int_as_float(0x7F800000) : E != 0 && q >= 1 ? f : 0.f;
}

// per-column exponents of a row-major R x C FP64 block (ex pre-set to kNoExp);
// SHIFT: of the block whose row r is scaled by 2^rexp[r]; SUMS: sum of |x| added per
// column.  A CTA takes 64 columns (two per thread, 32 threads) of `rows` rows (eight
// at a time); blockIdx.z: one of two blocks.  Without SHIFT the upper words decide
// (three integer instructions an entry where exp_bits takes a dozen; subnormal
// columns are read again).
struct ExpsArgs {
    const double *X;
    int C, ldx;
    bool vec;  // rows of 16-byte pairs
    int *ex;
    double *sums;
};
template <bool SHIFT, bool SUMS>
__global__ void __launch_bounds__(256) k_col_exps(int R, ExpsArgs p0, ExpsArgs p1, int rows, const int *__restrict__ rexp) {
    const ExpsArgs p = blockIdx.z ? p1 : p0;
    const double *__restrict__ X = p.X;
    const int C = p.C, ldx = p.ldx;
    const bool vec = p.vec;
    if ((int)blockIdx.y * 64 >= C) return;
    __shared__ int red[8][64];
    __shared__ double reds[SUMS ? 8 : 1][64];
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    const int j = blockIdx.y * 64 + 2 * tx;
    const int ra = blockIdx.x * rows + ty, r1 = min(R, (int)(blockIdx.x + 1) * rows);
    int m0 = kNoExp, m1 = kNoExp, ref0 = 0, ref1 = 0;
    unsigned h0 = 0, h1 = 0;
    float s0 = 0.f, s1 = 0.f;
#pragma unroll 4
    for (int r = ra; r < r1; r += 8) {
        const double *x = X + (size_t)r * ldx + j;
        double a = 0.0, b = 0.0;
        if (vec && j + 1 < C) {
            const double2 v = *reinterpret_cast<const double2 *>(x);
            a = v.x, b = v.y;
        } else {
            if (j < C) a = x[0];
            if (j + 1 < C) b = x[1];
        }
        if (SHIFT) {
            int ea = exp_bits(a), eb = exp_bits(b);
            const int q = rexp[r];
            if (ea != kNoExp) ea = ea == kNonFinite ? kBadExp : ea + q;
            if (eb != kNoExp) eb = eb == kNonFinite ? kBadExp : eb + q;
            m0 = max(m0, ea);
            m1 = max(m1, eb);
        } else {
            const unsigned ha = (unsigned)__double2hiint(a) & 0x7FFFFFFFu, hb = (unsigned)__double2hiint(b) & 0x7FFFFFFFu;
            h0 = max(h0, ha);
            h1 = max(h1, hb);
            if (SUMS) {
                add_abs(ha, ref0, s0);
                add_abs(hb, ref1, s1);
            }
        }
    }
    if (!SHIFT) {
        m0 = (int)(h0 >> 20) - 1022;
        m1 = (int)(h1 >> 20) - 1022;
        if (h0 < 0x100000u) {
            m0 = kNoExp;
            for (int r = ra; r < r1 && j < C; r += 8) m0 = max(m0, exp_bits(X[(size_t)r * ldx + j]));
        }
        if (h1 < 0x100000u) {
            m1 = kNoExp;
            for (int r = ra; r < r1 && j + 1 < C; r += 8) m1 = max(m1, exp_bits(X[(size_t)r * ldx + j + 1]));
        }
    }
    red[ty][2 * tx] = m0;
    red[ty][2 * tx + 1] = m1;
    if (SUMS) {
        reds[ty][2 * tx] = ldexp((double)s0, ref0 - 1023);
        reds[ty][2 * tx + 1] = ldexp((double)s1, ref1 - 1023);
    }
    __syncthreads();
    if (threadIdx.x < 64 && blockIdx.y * 64 + threadIdx.x < C) {
        int m = red[0][threadIdx.x];
#pragma unroll
        for (int q = 1; q < 8; ++q) m = max(m, red[q][threadIdx.x]);
        if (m != kNoExp) atomicMax(&p.ex[blockIdx.y * 64 + threadIdx.x], m);
        if (SUMS) {
            double t = reds[0][threadIdx.x];
#pragma unroll
            for (int q = 1; q < 8; ++q) t += reds[q][threadIdx.x];
            if (t != 0.0) atomicAdd(&p.sums[blockIdx.y * 64 + threadIdx.x], t);
        }
    }
}

// ---- which tiles of an FP64 product the seven digits may compute ----------------
//
// With |x| < 2^e per row of C (column of C), x = 2^e u, the digits leave
//     |error of C_ij| <= 2^(e_i + e_j) (2^-56 (sum |u_i| + sum |u_j|) + 2^-61 K),
// the rounding of either factor's last digit against the other factor, and the
// digit pairs left out.  FP64 arithmetic is held by sum |x_i| |x_j| instead (K
// 2^-53 of it in the worst case, a few 2^-53 as a rule), so an entry is left to the
// digits only where that sum is large enough:
//     sum |u_i| + sum |u_j| + K / 32 <= R h_ij,   h_ij = sum |u_i| |u_j|,
// R = min(8 K, 52 sqrt(K), 1024): K 2^-53 sum |x_i| |x_j| at the most if all K
// roundings had one sign, 2^-50 since they have either (sqrt(K) of them are felt).
// h is one BF16 product of the magnitudes, rounded down (a Gram takes every fourth
// or eighth row: part of the terms is a lower bound too).  The 64 x 64 tiles with an entry
// that fails, or with infinities or NaN, go to the FP64 kernel and are skipped here.
// Normal data have a left side of 0.2 to 0.3 K and a right side of 1.5 to 8 K; a
// second factor I + 0.3 N(0, 1) / sqrt(K) 42 to 72 and 190 to 370 at K = 300 (110 to
// 220 in the least of 49 million entries).  Columns graded from 1 to 10^-10
// against one that lives on the small half fail, where the digits left 2.4e-9 of
// sum |x_i| |x_j|.
static float digits_ratio(double k) { return (float)std::min({8.0 * k, 52.0 * std::sqrt(k), 1024.0}); }

// li, lj: entry_limit of sum |u_i| + K / 32 and of sum |u_j|
__device__ __forceinline__ bool digits_fail(float li, float lj, float ratio, float h) { return !(li + lj <= ratio * h); }

// tiles of an M x N Gram with entries that fail
__global__ void k_check_tiles(int M, int N, float k, float ratio, const float *__restrict__ h, const int *__restrict__ ex,
                              const double *__restrict__ sx, const int *__restrict__ ey, const double *__restrict__ sy,
                              int *__restrict__ tiles, int ntn) {
    const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (int64_t)M * N) return;
    const int i = (int)(idx / N), j = (int)(idx % N);
    const float li = entry_limit(ex[i], (float)ldexp(sx[i], -ex[i]) + k * 0.03125f);
    if (digits_fail(li, entry_limit(ey[j], (float)ldexp(sy[j], -ey[j])), ratio, h[idx]))
        tiles[(size_t)(i >> 6) * ntn + (j >> 6)] = 1;
}

// limits of n columns (sums |u| on entry) with their K / 32, up to np
__global__ void k_col_limits(int n, int np, float k, const int *__restrict__ ex, float *__restrict__ limits) {
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j < np) limits[j] = j < n ? entry_limit(ex[j], limits[j] + k * 0.03125f) : entry_limit(kNoExp, 0.f);
}

// Products whose result is held to norms instead (Rayleigh-Ritz): tiles with
// infinities or NaN and, with sums, columns i with K 2^e_i > 128 sum |x_i|, whose
// rounding to digits could pass 2^-48 ||x_i|| ||x_j||.  A CTA per tile.
__global__ void __launch_bounds__(128) k_guard_tiles(int M, int N, double k, const int *__restrict__ ex,
                                                     const double *__restrict__ sx, const int *__restrict__ ey,
                                                     const double *__restrict__ sy, int *__restrict__ tiles, int ntn) {
    const bool row = threadIdx.x < 64;
    const int i = (row ? blockIdx.x : blockIdx.y) * 64 + (threadIdx.x & 63);
    bool bad = false;
    if (i < (row ? M : N)) {
        const int e = (row ? ex : ey)[i];
        bad = bad_exp(e) || (sx && e != kNoExp && !(k <= 128.0 * ldexp((row ? sx : sy)[i], -e)));
    }
    if (__syncthreads_or(bad) && threadIdx.x == 0) tiles[(size_t)blockIdx.x * ntn + blockIdx.y] = 1;
}

// T + offset of x against the group exponent e (|x| < 2^e): T = round(x
// 2^(B-e)), B = 8 SL - 1, as an integer (|T| <= 2^B).  T in balanced base 256,
//     T = sum_s d_s 2^(8 (SL - 1 - s)),  d_1..d_{SL-1} in [-128, 127],  |d_0| <= 128,
// so x = 2^(e-7) sum_s d_s 2^(-8 s) up to 2^(e-B-1).  With 128 added at every
// digit below the top one, digit s + 128 is byte SL - 1 - s and d_0 is what
// stands above: no carry chain.
template <int SL>
__device__ __forceinline__ long long split_int(double x, int e) {
    const long long bits = __double_as_longlong(x);
    const int E = (int)((bits >> 52) & 0x7FF);
    const unsigned long long M = (bits & 0xFFFFFFFFFFFFFULL) | (E ? 1ULL << 52 : 0ULL);
    // x 2^(B-e) = +-M 2^sh, sh <= B - 53 <= 2 when |x| < 2^e, more for subnormals
    const int sh = (E ? E : 1) - 1075 + (8 * SL - 1) - e;
    unsigned long long t = (M << 3) >> min(max(2 - sh, 0), 63);
    if (sh > 2) t = M != 0 ? M << min(sh + 1, 63) : 0;
    const long long T = (long long)((t + 1) >> 1), neg = bits >> 63;
    constexpr long long off = (long long)(0x8080808080808080ULL >> (8 * (9 - SL)));
    return (T ^ neg) - neg + off;
}

// digits of the 8 values v[0..7] (consecutive k of one row, exponents e[.]) as
// one 16-byte vector per slice; out: the row's place in slice 0, slice_step:
// elements between slices.  Bytes become floats by placing them in the low
// mantissa of 2^23; a BF16 is the upper half of such an exact small float.
template <int SL>
__device__ __forceinline__ void split8_store(const double (&v)[8], const int (&e)[8], __nv_bfloat16 *out,
                                             size_t slice_step) {
    unsigned lo[8], hi[8];
#pragma unroll
    for (int t = 0; t < 8; ++t) {
        const long long T = split_int<SL>(v[t], e[t]);
        lo[t] = (unsigned)T;
        hi[t] = (unsigned)((unsigned long long)T >> 32);
    }
#pragma unroll
    for (int s = 0; s < SL; ++s) {
        unsigned w[4];
#pragma unroll
        for (int t = 0; t < 8; t += 2) {
            unsigned f[2];
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const int byte = SL - 1 - s;
                float x;
                if (s == 0)
                    x = __int_as_float(0x4B400000 + ((int)hi[t + u] >> (8 * (SL - 5)))) - 12582912.f;
                else
                    x = __uint_as_float(__byte_perm(byte < 4 ? lo[t + u] : hi[t + u], 0x4B000000u, 0x7440u | (byte & 3))) -
                        8388736.f;
                f[u] = __float_as_uint(x);
            }
            w[t / 2] = __byte_perm(f[0], f[1], 0x7632);
        }
        *reinterpret_cast<uint4 *>(out + s * slice_step) = make_uint4(w[0], w[1], w[2], w[3]);
    }
}

// one slice of magnitudes: u = |v| 2^-e as BF16, rounded down
template <>
__device__ __forceinline__ void split8_store<1>(const double (&v)[8], const int (&e)[8], __nv_bfloat16 *out, size_t) {
    unsigned w[4];
#pragma unroll
    for (int t = 0; t < 8; t += 2)
        w[t / 2] = __byte_perm(__float_as_uint(scaled_abs(v[t], e[t])), __float_as_uint(scaled_abs(v[t + 1], e[t + 1])), 0x7632);
    *reinterpret_cast<uint4 *>(out) = make_uint4(w[0], w[1], w[2], w[3]);
}

// Global layout of the digit slices: for K step kc = k / 16, row block b = r /
// RB (RB = 128 rows for the first operand of a product, 64 for the second) and
// slice s, the 8 x 8 core matrices (8 rows x 16 bytes) of the RB x 16 block in
// the order [r % RB / 8][k % 16 / 8], blocks ordered [kc][b][s]: all slices of
// one product tile and K step are one contiguous piece.
template <int SL>
__device__ __forceinline__ size_t tiled_off(int r, int k, int nb, int rb_log) {
    const int b = r >> rb_log, rr = r & ((1 << rb_log) - 1);
    return ((((size_t)(k >> 4) * nb + b) * SL) << (rb_log + 4)) + (size_t)(rr >> 3) * 128 + (size_t)((k >> 3) & 1) * 64 +
           (size_t)(rr & 7) * 8;
}

// split a row-major R x K block per row (K = columns): one thread per row and
// 8-wide K group; a warp covers one 8-row group x 32 columns.  cexp: column k
// of the block is scaled by 2^-cexp[k] before the split; mags (may be null): the
// slice of magnitudes as well.
template <int SL>
__global__ void __launch_bounds__(256) k_split_rows(int R, int K, const double *__restrict__ X, int ldx, bool vec,
                                                    const int *__restrict__ ex, const int *__restrict__ cexp,
                                                    __nv_bfloat16 *__restrict__ out, int rows_p, int kp, int rb_log,
                                                    __nv_bfloat16 *__restrict__ mags) {
    const int64_t gw = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    const int KC = (kp + 31) / 32;
    if (gw >= (int64_t)(rows_p / 8) * KC) return;
    const int rg = (int)(gw / KC), kc = (int)(gw % KC);
    const int r = rg * 8 + (lane & 7), k0 = kc * 32 + (lane >> 3) * 8;
    if (k0 >= kp) return;
    double v[8];
    int e[8];
    const double *x = X + (size_t)r * ldx + k0;
    if (vec && r < R && k0 + 8 <= K) {
#pragma unroll
        for (int t = 0; t < 8; t += 2) {
            const double2 q = *reinterpret_cast<const double2 *>(x + t);
            v[t] = q.x, v[t + 1] = q.y;
        }
    } else {
#pragma unroll
        for (int t = 0; t < 8; ++t) v[t] = (r < R && k0 + t < K) ? x[t] : 0.0;
    }
    const int er = r < R ? ex[r] : kNoExp;
#pragma unroll
    for (int t = 0; t < 8; ++t) e[t] = er + (cexp && k0 + t < K ? cexp[k0 + t] : 0);
    split8_store<SL>(v, e, out + tiled_off<SL>(r, k0, rows_p >> rb_log, rb_log), (size_t)16 << rb_log);
    if (SL == 7 && mags) split8_store<1>(v, e, mags + tiled_off<1>(r, k0, rows_p >> rb_log, rb_log), 0);
}

// split a row-major K x C block per column (operand row r = column r, K = rows
// of X), transposed through shared memory: a block handles 64 columns and `tiles`
// times 32 K rows, two tiles on their way (cp.async) while one is split; half a
// warp reads 16 columns of eight rows, a warp stores 512 contiguous bytes.
// rexp: row k of the block is scaled by 2^rexp[k].  sums (magnitudes, SL = 1): the
// sum over k of u added per column.
// What bounds it: memory (a 250,000 x 750 block into five digits: 0.55 ms,
// 6.1 TB/s; a tile per block through registers 0.75 ms, waiting for its loads).
constexpr int kSplitPitch = 66;                         // doubles: 16-byte rows
constexpr int kSplitSmem = 3 * 32 * kSplitPitch * 8;    // three tiles
// blockIdx.z: one of two blocks.
struct SplitArgs {
    const double *X;
    int C, ldx;
    bool vec;  // rows of 16-byte pairs
    const int *ex;
    __nv_bfloat16 *out;
    int rows_p, rb_log;
};
template <int SL>
__global__ void __launch_bounds__(256, 4) k_split_cols(int K, SplitArgs p0, SplitArgs p1, const int *__restrict__ rexp,
                                                       int kp, float *__restrict__ sums, int tiles) {
    extern __shared__ __align__(16) double tile[];
    const SplitArgs p = blockIdx.z ? p1 : p0;
    const double *__restrict__ X = p.X;
    const int C = p.C, ldx = p.ldx, rows_p = p.rows_p, rb_log = p.rb_log;
    const bool vec = p.vec;
    if ((int)blockIdx.y * 64 >= rows_p) return;
    const int c0 = blockIdx.y * 64, t0 = blockIdx.x * tiles, t1 = min(t0 + tiles, (kp + 31) / 32);
    auto stage = [&](int t) {
        if (t < t1) {
            double *dst = tile + (size_t)((t - t0) % 3) * 32 * kSplitPitch;
            // rows past K and columns past C: zeros (no byte read)
            if (vec) {
#pragma unroll
                for (int q = threadIdx.x; q < 1024; q += 256) {
                    const int yy = q >> 5, c = 2 * (q & 31), k = 32 * t + yy;
                    const int bytes = k < K ? 8 * max(0, min(2, C - c0 - c)) : 0;
                    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(
                                     (unsigned)__cvta_generic_to_shared(dst + yy * kSplitPitch + c)),
                                 "l"(bytes ? X + (size_t)k * ldx + c0 + c : X), "r"(bytes));
                }
            } else {
#pragma unroll
                for (int q = threadIdx.x; q < 2048; q += 256) {
                    const int yy = q >> 6, c = q & 63, k = 32 * t + yy;
                    const int bytes = k < K && c0 + c < C ? 8 : 0;
                    asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;\n" ::"r"(
                                     (unsigned)__cvta_generic_to_shared(dst + yy * kSplitPitch + c)),
                                 "l"(bytes ? X + (size_t)k * ldx + c0 + c : X), "r"(bytes));
                }
            }
        }
        asm volatile("cp.async.commit_group;\n" ::: "memory");
    };
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int lc = (lane & 15) + 16 * (wid & 3), kg = (lane >> 4) + 2 * (wid >> 2), r = c0 + lc;
    const int er = r < C ? p.ex[r] : kNoExp;
    float ss = 0.f;
    stage(t0);
    stage(t0 + 1);
    for (int t = t0; t < t1; ++t) {
        asm volatile("cp.async.wait_group 1;\n" ::: "memory");
        __syncthreads();  // tile t is there, the one of t - 1 is free
        stage(t + 2);
        const double *src = tile + (size_t)((t - t0) % 3) * 32 * kSplitPitch + kg * 8 * kSplitPitch + lc;
        const int k = 32 * t + 8 * kg;
        double v[8];
        int e[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            v[u] = src[u * kSplitPitch];
            e[u] = er - (rexp && k + u < K ? rexp[k + u] : 0);
        }
        if (r < rows_p && k < kp)
            split8_store<SL>(v, e, p.out + tiled_off<SL>(r, k, rows_p >> rb_log, rb_log), (size_t)16 << rb_log);
        if (SL == 1 && sums) {
#pragma unroll
            for (int u = 0; u < 8; ++u) ss += scaled_abs(v[u], e[u]);
        }
    }
    if (SL == 1 && sums) {
        ss += __shfl_xor_sync(0xffffffffu, ss, 16);
        if (lane < 16 && r < C && ss > 0.f) atomicAdd(&sums[r], ss);
    }
}

__global__ void k_fill_int(int n, int v, int *__restrict__ x) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) x[i] = v;
}

__device__ __forceinline__ unsigned smem_addr(const void *p) {
    return (unsigned)__cvta_generic_to_shared(p);
}

// SMs of the current device (queried per call: a process may drive GPUs of
// different sizes; the attribute query costs about a microsecond)
int sm_count_oz() {
    int dev = 0, c = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&c, cudaDevAttrMultiProcessorCount, dev);
    return c > 0 ? c : 1;
}

// ---- the product kernel (tcgen05, TMEM) --------------------------------------
//
// Work item: a 128 x 64 tile of C over a range of K; a persistent CTA per SM
// takes the items blockIdx.x, blockIdx.x + gridDim.x, ...  K is staged 16 deep
// through a ring of shared-memory stages by bulk copies (TMA, cp.async.bulk):
// the operand layout keeps all digit slices of one tile and K step contiguous,
// so a stage is two copies, landing in core-matrix order [s][r/8][k/8][8 x 16
// bytes] (LBO = 128 bytes between K groups, SBO = 256 bytes between 8-row
// groups).  Because the Y slices of a stage follow each other at the row-group
// stride, [Y_0 .. Y_{w-1}] is one N = 64 w operand: one MMA (two above N = 256)
// multiplies X_s by [Y_0 .. Y_{w-1}], w = min(SL, ND - s), and its 64-column
// blocks land on the accumulators acc_s .. acc_{s+w-1} of the digit sums D = s +
// t, which sit side by side in TMEM (ND x 64 columns).
//
// Exactness: a digit product is at most 2^14 in magnitude, and the sum for D
// takes D + 1 pairs per K row, so after kChunk = 256 rows the sums for D <= 3
// are at most 2^24 and exact in FP32.  A sum for D >= 4 (weight 2^-32 and less)
// can pass 2^24, and each MMA after that may round it by a unit.  For D = 4 and 5
// that takes digits of one sign and nearly full size in all D + 1 pairs, those of the
// leading digits among them: four pairs alone stay within 2^24.  With the leading
// digit of the smaller factor at r of its full size, at most r / 4 of the chunk's
// 80 (D = 4) MMAs come after, 20 r units of 2^-46 of the maxima's product next to
// 190 r of that product in sum |x| |y|: 2^-49 of it at the worst.  From D = 6 on the
// units weigh 2^-62 and less.  Every chunk is drained into FP32 expansions in
// registers.
//
// The drain stops the tensor cores briefly: the accumulators of the highest D
// (three of five digits' sums, two of six digits') have two sets of TMEM
// columns that alternate from chunk to chunk, and the first step of a chunk is
// issued in descending slices: those that touch only the alternating
// accumulators at once, the others as the drain releases theirs (seven digits
// fill TMEM with one set).  An accumulator's first MMA of a chunk overwrites it
// (its own N = 64 instruction).  Starting more steps of a chunk this way was
// slower (2.70 ms with three, 2.54 with one, 250,000 x 750 x 750, five digits):
// the stages that it holds come back late.
//
// What bounds it: a Gram of 250,000 x 750 x 750 takes 2.5 / 3.7 / 5.7 ms with
// five, six and seven digits; the MMAs alone (no loads, no drain) take 2.08 /
// 2.88 / 4.48, with the loads 2.29 / 3.18 / 4.82, the rest is the drain.  One CTA
// per tile, K staged 32 deep in twelve copies, one set of accumulators and MMAs
// issued by a lone lane: 3.53 ms with five digits; the update of the same sizes
// (six digits, 23,448 tiles 47 steps deep) 6.43 ms, now 3.7.
//
// Warp roles (320 threads): warp 0 issues the loads, warp 1 owns TMEM and
// issues the MMAs (one thread), warps 2..9 drain, one TMEM lane (output row)
// and 32 of the 64 columns per thread, and write the item's results while the
// MMAs of the next item run.  Every mbarrier wait gives up after 2 s, records that
// in the caller's error word, which the host checks, and the CTA still drains its own copies
// and MMAs and frees its TMEM.
// ------------------------------------------------------------------------------
constexpr int TC_M = 128, TC_N = 64, TC_K = 16;
constexpr int TC_THREADS = 320, TC_DRAIN_WARPS = 8;
constexpr int kChunk = 256;                 // K rows per drained chunk
constexpr int kChunkSteps = kChunk / TC_K;  // 16
// K rows of one work item at most: the low word of the FP32 expansions takes
// one rounding per chunk, 64 of them stay below the digits' own truncation;
// longer products add their items in FP64
constexpr int kItemK = 16384;
// digit sums kept: pairs with s + t >= ND are dropped
template <int SL> __host__ __device__ constexpr int tc_nd() { return SL == 7 ? 8 : SL; }
template <int SL> __host__ __device__ constexpr uint32_t tc_a_bytes() { return 2u * TC_M * TC_K * SL; }
template <int SL> __host__ __device__ constexpr uint32_t tc_b_bytes() { return 2u * TC_N * TC_K * SL; }
template <int SL> __host__ __device__ constexpr uint32_t tc_stage_bytes() { return tc_a_bytes<SL>() + tc_b_bytes<SL>(); }
// stages that fit 220 KB: 7, 6, 5 for 5, 6, 7 digits
template <int SL> __host__ __device__ constexpr int tc_stages() { return (int)(220u * 1024u / tc_stage_bytes<SL>()); }
// accumulators with one set of columns; the ND - tc_low above them have two
template <int SL> __host__ __device__ constexpr int tc_low() { return SL == 5 ? 2 : SL == 6 ? 4 : 8; }
template <int SL> constexpr size_t tc_smem() { return (size_t)tc_stages<SL>() * tc_stage_bytes<SL>() + 1024; }
constexpr uint32_t TC_TMEM_COLS = 512;
constexpr uint64_t TC_WAIT_NS = 2000000000ull;  // 2 s per barrier wait

// shared-memory matrix descriptor, low word: start >> 4 (bits 0-13), LBO >> 4
// (16-29); high word: SBO >> 4 (32-45), descriptor version 1 (46-47), no
// swizzle (61-63 = 0).  Addresses stay below 2^18, so offsets are added to the
// low word as they are.
__device__ __forceinline__ uint32_t umma_desc_lo(uint32_t saddr, uint32_t lbo) { return (saddr >> 4) | ((lbo >> 4) << 16); }
__device__ __forceinline__ uint64_t umma_desc(uint32_t lo, uint32_t sbo) {
    return ((uint64_t)((sbo >> 4) | (1u << 14)) << 32) | lo;
}

// instruction descriptor of kind::f16: FP32 accumulator, BF16 A and B, both
// K-major, N >> 3 at bit 17, M >> 4 at bit 24
__host__ __device__ constexpr uint32_t umma_idesc(int m, int n) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(m >> 4) << 24);
}

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(bar), "r"(count));
}

__device__ __forceinline__ uint64_t global_ns() {
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;\n" : "=l"(t));
    return t;
}

// wait for the phase of the given parity; gives up after TC_WAIT_NS of wall time
// and sets *err
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, int *err) {
    uint64_t t0 = 0;
    for (uint32_t it = 0;; ++it) {
        uint32_t ok;
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(ok)
            : "r"(bar), "r"(parity)
            : "memory");
        if (ok) return true;
        if ((it & 255u) == 0) {
            const uint64_t t = global_ns();
            if (it == 0) t0 = t;
            else if (t - t0 > TC_WAIT_NS) break;
        }
    }
    atomicExch(err, 1);
    return false;
}

__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(bar) : "memory");
}

// bulk copy (TMA) of `bytes` contiguous bytes global -> shared, completing on bar
__device__ __forceinline__ void bulk_load(uint32_t dst, const void *src, uint32_t bytes, uint32_t bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(dst),
                 "l"(reinterpret_cast<uint64_t>(src)), "r"(bytes), "r"(bar)
                 : "memory");
}

// one lane of a converged warp
__device__ __forceinline__ uint32_t elect_lane() {
    uint32_t p;
    asm volatile("{\n .reg .pred q;\n elect.sync _|q, 0xffffffff;\n selp.u32 %0, 1, 0, q;\n}\n" : "=r"(p));
    return p;
}

// Issued by the elected lane of a converged warp: operands that are the same
// in the whole warp stay in uniform registers, which the instruction takes (48
// clocks per small MMA; 118 when one lane runs the loop alone and every operand
// is moved over, more than a 128 x 64 x 16 product's 32)
__device__ __forceinline__ void umma_f16(uint32_t dtmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc, int acc,
                                         uint32_t el) {
    asm volatile(
        "{\n .reg .pred p, q;\n setp.ne.b32 p, %4, 0;\n setp.ne.b32 q, %5, 0;\n"
        " @q tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(dtmem),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(acc), "r"(el));
}

__device__ __forceinline__ void umma_commit(uint32_t bar, uint32_t el) {
    asm volatile(
        "{\n .reg .pred q;\n setp.ne.b32 q, %1, 0;\n"
        " @q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n}\n" ::"r"(bar),
        "r"(el)
        : "memory");
}

// n consecutive 32-bit TMEM columns of the warp's 32 lanes (one lane per
// thread); the registers may be read after tmem_wait on them (which waits for
// every load issued before it)
template <int n> __device__ __forceinline__ void tmem_ld(uint32_t taddr, uint32_t (&r)[n]);
template <int n> __device__ __forceinline__ void tmem_wait(uint32_t (&r)[n]);
template <>
__device__ __forceinline__ void tmem_ld<32>(uint32_t taddr, uint32_t (&r)[32]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
                 : "r"(taddr));
}
template <>
__device__ __forceinline__ void tmem_wait<32>(uint32_t (&r)[32]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;\n" : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]), "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15]), "+r"(r[16]), "+r"(r[17]), "+r"(r[18]), "+r"(r[19]), "+r"(r[20]), "+r"(r[21]), "+r"(r[22]), "+r"(r[23]), "+r"(r[24]), "+r"(r[25]), "+r"(r[26]), "+r"(r[27]), "+r"(r[28]), "+r"(r[29]), "+r"(r[30]), "+r"(r[31])::"memory");
}
template <>
__device__ __forceinline__ void tmem_ld<8>(uint32_t taddr, uint32_t (&r)[8]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr));
}
template <>
__device__ __forceinline__ void tmem_wait<8>(uint32_t (&r)[8]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;\n" : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7])::"memory");
}

// s = fl(a + b), returns the rounding error a + b - s exactly (Knuth)
__device__ __forceinline__ float two_sum(float a, float b, float &s) {
    s = __fadd_rn(a, b);
    const float bp = __fsub_rn(s, a);
    return __fadd_rn(__fsub_rn(a, __fsub_rn(s, bp)), __fsub_rn(b, bp));
}

// One chunk's digit sums of a value added into its expansion.  In units of the
// D = 0 sum the chunk is r0 + 2^-8 r1 + 2^-16 r2 + 2^-24 v, r0..r2 integers
// below 2^24.  s = fl(r0 + 2^-8 r1) with the exact remainder, to which 2^-16 r2
// adds exactly (multiples of 2^-16 below 2^8): error-free terms for hi; the
// errors go to lo.  v, the digits from D = 3 on, goes to lo too with five
// digits; with six, whose dropped pairs weigh 2^-48, its rounding and lo's would
// be felt (0.1 of the error at K = 750): it comes with its own error ev and is
// the third term for hi.
template <int SL>
__device__ __forceinline__ void add_chunk(float r0, float r1, float r2, float v, float ev, float &hi, float &lo) {
    const float s = __fmaf_rn(r1, 0x1p-8f, r0);
    const float e = __fmaf_rn(r1, 0x1p-8f, __fsub_rn(r0, s));
    const float t = __fmaf_rn(r2, 0x1p-16f, e);
    float h;
    const float e1 = two_sum(hi, s, h);
    if constexpr (SL == 5) {
        const float e2 = two_sum(h, t, hi);
        lo = __fmaf_rn(v, 0x1p-24f, __fadd_rn(lo, __fadd_rn(e1, e2)));
    } else {
        float h2;
        const float e2 = two_sum(h, t, h2);
        const float e3 = two_sum(h2, __fmul_rn(v, 0x1p-24f), hi);
        lo = __fadd_rn(lo, __fadd_rn(__fadd_rn(e1, e2), __fmaf_rn(ev, 0x1p-24f, e3)));
    }
}

// the same for seven digits, into three words: 2^-24 (s3 + f3) replaces v
__device__ __forceinline__ void add_chunk3(float r0, float r1, float r2, float s3, float f3, float &hi, float &mid,
                                           float &lo) {
    const float s = __fmaf_rn(r1, 0x1p-8f, r0);
    const float e = __fmaf_rn(r1, 0x1p-8f, __fsub_rn(r0, s));
    const float t = __fmaf_rn(r2, 0x1p-16f, e);
    float p, h, m;
    const float pe = two_sum(t, __fmul_rn(s3, 0x1p-24f), p);
    const float e1 = two_sum(hi, s, h);
    hi = h;
    const float e2 = two_sum(mid, e1, m);
    const float e3 = two_sum(m, p, mid);
    lo = __fadd_rn(lo, __fadd_rn(__fadd_rn(e2, e3), __fmaf_rn(f3, 0x1p-24f, pe)));
}

// exact FP32 -> FP64 of zero and normal numbers (the digit sums are multiples of
// 2^-48: no subnormals)
__device__ __forceinline__ double f2d_normal(float x) {
    const unsigned u = __float_as_uint(x);
    const unsigned h = (u & 0x80000000u) | (((u >> 3) & 0x0FFFFFFFu) + 0x38000000u);
    return __hiloint2double((int)(x == 0.f ? 0u : h), (int)(x == 0.f ? 0u : u << 29));
}

// Work items of one product (host-built, passed by value)
struct TcWork {
    int ntn, tiles, items;  // column tiles, output tiles, tiles x K ranges
    int ksteps, split;      // K steps of the product, K steps per item
    int lower;              // tiles meeting the lower triangle only
    const int *skip;        // 64 x 64 tiles left to others (nonzero), skip_ld to a row of tiles; may be null
    int skip_ld;
};
struct TcItem {
    int i0, j0, kc0, nk;
};
__device__ __forceinline__ TcItem tc_item(const TcWork &w, int item) {
    const int sp = item / w.tiles, tile = item - sp * w.tiles;
    int ti, tj;
    if (w.lower) {  // row tile ti meets the column tiles 0 .. 2 ti + 1 (at most ntn)
        ti = 0;
        int left = tile;
        for (int c = min(2, w.ntn); left >= c; c = min(2 * ti + 2, w.ntn)) {
            left -= c;
            ++ti;
        }
        tj = left;
    } else {
        ti = tile / w.ntn;
        tj = tile - ti * w.ntn;
    }
    TcItem it;
    it.i0 = ti * TC_M;
    it.j0 = tj * TC_N;
    it.kc0 = sp * w.split;
    it.nk = min(w.split, w.ksteps - it.kc0);
    return it;
}

// whether one of the item's two 64 x 64 tiles is wanted
__device__ __forceinline__ bool tc_wanted(const TcWork &w, const TcItem &it, int M) {
    if (!w.skip) return true;
    const int c = it.j0 / 64;
    bool wanted = false;
    for (int q = it.i0 / 64; q < it.i0 / 64 + 2; ++q)
        wanted |= q * 64 < M && !(w.lower && c > q) && w.skip[(size_t)q * w.skip_ld + c] == 0;
    return wanted;
}

template <int SL>
__global__ void __launch_bounds__(TC_THREADS, 1)
    k_ozaki_tc(int M, int N, const __nv_bfloat16 *__restrict__ Xs, int nbx, const __nv_bfloat16 *__restrict__ Ys,
               int nby, const int *__restrict__ ex, const int *__restrict__ ey, double *__restrict__ C, int ldc,
               TcWork w, int atomic, int vec, int *__restrict__ err) {
    constexpr int ND = tc_nd<SL>(), STAGES = tc_stages<SL>(), LOW = tc_low<SL>();
    constexpr uint32_t A_BYTES = tc_a_bytes<SL>(), B_BYTES = tc_b_bytes<SL>(), STAGE = tc_stage_bytes<SL>();
    constexpr uint32_t LBO = 128, SBO = 256, SLICE_A = A_BYTES / SL, SLICE_B = B_BYTES / SL;
    extern __shared__ unsigned char smem_dyn[];
    // accf: a chunk is complete; free_bar: its low accumulators are drained (two
    // groups with six digits); high_bar: all of it is
    __shared__ __align__(8) uint64_t full_bar[STAGES], empty_bar[STAGES], accf_bar, free_bar[2], high_bar, drain_bar;
    __shared__ uint32_t tmem_slot;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // stages on a 1024-byte boundary
    const uint32_t smem0 = (smem_addr(smem_dyn) + 1023u) & ~1023u;
    if (threadIdx.x == 0) {
        for (int st = 0; st < STAGES; ++st) {
            mbar_init(smem_addr(&full_bar[st]), 1);
            mbar_init(smem_addr(&empty_bar[st]), 1);
        }
        mbar_init(smem_addr(&accf_bar), 1);
        mbar_init(smem_addr(&free_bar[0]), TC_DRAIN_WARPS);
        mbar_init(smem_addr(&free_bar[1]), TC_DRAIN_WARPS);
        mbar_init(smem_addr(&high_bar), TC_DRAIN_WARPS);
        mbar_init(smem_addr(&drain_bar), 1);
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_addr(&tmem_slot)),
                     "r"(TC_TMEM_COLS));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n");
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    const uint32_t tmem = tmem_slot;

    if (warp == 0) {
        if (lane == 0) {
            // producer: a stage is refilled once the MMAs of its previous step completed
            bool ok = true;
            int g = 0;  // K steps issued by this CTA so far
            for (int item = blockIdx.x; item < w.items && ok; item += gridDim.x) {
                const TcItem it = tc_item(w, item);
                if (!tc_wanted(w, it, M)) continue;
                const __nv_bfloat16 *xa = Xs + ((size_t)it.kc0 * nbx + it.i0 / TC_M) * (A_BYTES / 2);
                const __nv_bfloat16 *yb = Ys + ((size_t)it.kc0 * nby + it.j0 / TC_N) * (B_BYTES / 2);
                for (int kt = 0; kt < it.nk; ++kt, ++g) {
                    const int st = g % STAGES;
                    if (g >= STAGES) ok = mbar_wait(smem_addr(&empty_bar[st]), ((g / STAGES) & 1) ^ 1, err);
                    if (!ok) break;
                    const uint32_t fb = smem_addr(&full_bar[st]), dst = smem0 + st * STAGE;
                    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(fb), "r"(STAGE)
                                 : "memory");
                    bulk_load(dst, xa + (size_t)kt * nbx * (A_BYTES / 2), A_BYTES, fb);
                    bulk_load(dst + A_BYTES, yb + (size_t)kt * nby * (B_BYTES / 2), B_BYTES, fb);
                }
            }
            // the last loads of every stage have landed before the CTA exits
            for (int q = max(0, g - STAGES); q < g; ++q) mbar_wait(smem_addr(&full_bar[q % STAGES]), (q / STAGES) & 1, err);
        }
    } else if (warp == 1) {
        // the whole warp runs the loop, the elected lane issues
        const uint32_t el = elect_lane();
        const uint32_t d0 = umma_desc_lo(smem0, LBO), full0 = smem_addr(full_bar), empty0 = smem_addr(empty_bar);
        // the digit sums D in [da, db] of slice sl: X_sl by [Y_{da-sl} .. Y_{db-sl}] of the
        // stage at descriptor word dw onto acc_da .. acc_db (all below LOW or
        // all from LOW on; hi: first column of the alternating set, less 64 LOW)
        auto part = [&](uint32_t dw, uint32_t hi, int sl, int da, int db, int acc) {
            const uint64_t ad = umma_desc(dw + ((sl * SLICE_A) >> 4), SBO);
            const uint32_t b = dw + ((A_BYTES + (da - sl) * SLICE_B) >> 4), d = (da < LOW ? tmem : hi) + TC_N * da;
            const int n = TC_N * (db - da + 1), n1 = n > 256 ? n / 2 : n;
            umma_f16(d, ad, umma_desc(b, SBO), umma_idesc(TC_M, n1), acc, el);
            if (n > 256)
                umma_f16(d + n1, ad, umma_desc(b + (((uint32_t)(n1 / 8) * SBO) >> 4), SBO), umma_idesc(TC_M, n1), acc, el);
        };
        // all digit sums of slice sl from da on
        auto slice = [&](uint32_t dw, uint32_t hi, int sl, int da) {
            const int db = (sl + SL - 1 < ND - 1 ? sl + SL - 1 : ND - 1);
            if (da > db) return;
            if (da < LOW && db >= LOW) {
                part(dw, hi, sl, da, LOW - 1, 1);
                part(dw, hi, sl, LOW, db, 1);
            } else {
                part(dw, hi, sl, da, db, 1);
            }
        };
        bool ok = true;
        uint32_t st = 0, ph = 0, c = 0;  // stage and its parity, chunks started by this CTA
        for (int item = blockIdx.x; item < w.items && ok; item += gridDim.x) {
            const TcItem it = tc_item(w, item);
            if (!tc_wanted(w, it, M)) continue;
            const int nk = it.nk;
            for (int k0 = 0; k0 < nk && ok; k0 += kChunkSteps, ++c) {
                const int steps = min(kChunkSteps, nk - k0);
                const uint32_t ap = (c - 1) & 1;  // parity of the chunk before
                const uint32_t hi = tmem + (c & 1) * TC_N * (ND - LOW);
                // first step of the chunk: every accumulator is overwritten once
                ok = mbar_wait(full0 + 8 * st, ph, err);
                const uint32_t dw = d0 + st * (STAGE >> 4);
                if constexpr (SL == 7) {
                    if (c > 0) ok = ok && mbar_wait(smem_addr(&free_bar[0]), ap, err);
                    if (!ok) break;
                    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
                    part(dw, hi, 0, 0, 6, 0);  // acc_0 .. acc_6 start
                    part(dw, hi, 1, 7, 7, 0);  // acc_7 starts
                    part(dw, hi, 1, 1, 6, 1);
#pragma unroll
                    for (int sl = 2; sl < 7; ++sl) slice(dw, hi, sl, sl);
                } else {
#pragma unroll
                    for (int sl = SL - 1; sl >= 0; --sl) {
                        // the alternating set is free since the chunk before
                        // ended, acc_3 and acc_2 (six digits), acc_1 and acc_0
                        // when the drain says so
                        if (c > 0 && (sl == 1 || (SL == 6 && sl == 3))) {
                            ok = ok && mbar_wait(smem_addr(&free_bar[SL == 6 && sl == 1 ? 1 : 0]), ap, err);
                            asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
                        }
                        if (!ok) break;
                        part(dw, hi, sl, sl, sl, 0);
                        slice(dw, hi, sl, sl + 1);
                    }
                }
                if (!ok) break;
                umma_commit(empty0 + 8 * st, el);
                if (++st == STAGES) st = 0, ph ^= 1;
                for (int q = 1; q < steps; ++q) {
                    ok = mbar_wait(full0 + 8 * st, ph, err);
                    if (!ok) break;
                    const uint32_t dw = d0 + st * (STAGE >> 4);
#pragma unroll
                    for (int sl = 0; sl < SL; ++sl) slice(dw, hi, sl, sl);
                    umma_commit(empty0 + 8 * st, el);
                    if (++st == STAGES) st = 0, ph ^= 1;
                }
                // the other alternating set, which the next chunk starts on, is
                // drained (waited for here, before this chunk's own completion,
                // so that the barrier is never two phases ahead)
                if (SL != 7 && c > 0) {
                    ok = ok && mbar_wait(smem_addr(&high_bar), ap, err);
                    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
                }
                if (!ok) break;
                umma_commit(smem_addr(&accf_bar), el);
            }
        }
        // every MMA issued by this warp has completed before teardown
        umma_commit(smem_addr(&drain_bar), el);
        mbar_wait(smem_addr(&drain_bar), 0, err);
    } else {
        // drain warps: TMEM lane quadrant = warp % 4, one output row and one
        // 32-column half per thread
        const int quad = warp & 3, c0 = 32 * ((warp - 2) >> 2);
        const uint32_t tbase = tmem + ((uint32_t)(32 * quad) << 16) + c0;
        auto release = [&](uint64_t &bar) {
            asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_addr(&bar));
        };
        auto f = [](uint32_t x) { return __uint_as_float(x); };
        bool ok = true;
        int c = 0;
        for (int item = blockIdx.x; item < w.items && ok; item += gridDim.x) {
            const TcItem it = tc_item(w, item);
            if (!tc_wanted(w, it, M)) continue;
            float hi[32], lo[32], mid[SL == 7 ? 32 : 1];
#pragma unroll
            for (int q = 0; q < 32; ++q) hi[q] = lo[q] = 0.f;
            if constexpr (SL == 7)
#pragma unroll
                for (int q = 0; q < 32; ++q) mid[q] = 0.f;
            const int nchunks = (it.nk + kChunkSteps - 1) / kChunkSteps;
            for (int ch = 0; ch < nchunks && ok; ++ch, ++c) {
                ok = __all_sync(0xffffffffu, mbar_wait(smem_addr(&accf_bar), c & 1, err));
                if (!ok) break;
                asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
                const uint32_t thigh = tbase + (c & 1) * TC_N * (ND - LOW);
                if constexpr (SL == 7) {
                    // 8 columns at a time (registers); the accumulators are
                    // released with the last of them
#pragma unroll
                    for (int h = 0; h < 4; ++h) {
                        uint32_t ra[8], rb[8];
                        float s4[8], s3[8], f3[8];
                        tmem_ld<8>(tbase + 8 * h + TC_N * 7, ra);
                        tmem_ld<8>(tbase + 8 * h + TC_N * 6, rb);
                        tmem_wait<8>(ra);
                        tmem_wait<8>(rb);
#pragma unroll
                        for (int q = 0; q < 8; ++q) s4[q] = __fmaf_rn(f(ra[q]), 0x1p-8f, f(rb[q]));
                        tmem_ld<8>(tbase + 8 * h + TC_N * 5, ra);
                        tmem_ld<8>(tbase + 8 * h + TC_N * 4, rb);
                        tmem_wait<8>(ra);
                        tmem_wait<8>(rb);
#pragma unroll
                        for (int q = 0; q < 8; ++q) {
                            const float g = __fmaf_rn(s4[q], 0x1p-8f, f(ra[q])), x = f(rb[q]);
                            s4[q] = __fmaf_rn(g, 0x1p-8f, x);
                            f3[q] = __fmaf_rn(g, 0x1p-8f, __fsub_rn(x, s4[q]));
                        }
                        uint32_t rc[8];
                        tmem_ld<8>(tbase + 8 * h + TC_N * 3, ra);
                        tmem_wait<8>(ra);
#pragma unroll
                        for (int q = 0; q < 8; ++q) {
                            const float e = two_sum(f(ra[q]), __fmul_rn(s4[q], 0x1p-8f), s3[q]);
                            f3[q] = __fmaf_rn(f3[q], 0x1p-8f, e);
                        }
                        tmem_ld<8>(tbase + 8 * h + TC_N * 2, rc);
                        tmem_ld<8>(tbase + 8 * h + TC_N, rb);
                        tmem_ld<8>(tbase + 8 * h, ra);
                        tmem_wait<8>(rc);
                        tmem_wait<8>(rb);
                        tmem_wait<8>(ra);
                        if (h == 3) release(free_bar[0]);
#pragma unroll
                        for (int q = 0; q < 8; ++q)
                            add_chunk3(f(ra[q]), f(rb[q]), f(rc[q]), s3[q], f3[q], hi[8 * h + q], mid[8 * h + q],
                                       lo[8 * h + q]);
                    }
                } else if constexpr (SL == 6) {
                    // acc_3 and acc_2 first, then 8 columns at a time
                    uint32_t r3[32], r2[32];
                    tmem_ld<32>(tbase + TC_N * 3, r3);
                    tmem_ld<32>(tbase + TC_N * 2, r2);
                    tmem_wait<32>(r3);
                    tmem_wait<32>(r2);
                    release(free_bar[0]);
#pragma unroll
                    for (int h = 0; h < 4; ++h) {
                        uint32_t ra[8], rb[8];
                        float v[8], ev[8];
                        tmem_ld<8>(thigh + 8 * h + TC_N * 5, ra);
                        tmem_ld<8>(thigh + 8 * h + TC_N * 4, rb);
                        tmem_wait<8>(ra);
                        tmem_wait<8>(rb);
#pragma unroll
                        for (int q = 0; q < 8; ++q) {
                            const float g = __fmaf_rn(f(ra[q]), 0x1p-8f, f(rb[q])), x = f(r3[8 * h + q]);
                            v[q] = __fmaf_rn(g, 0x1p-8f, x);
                            ev[q] = __fmaf_rn(g, 0x1p-8f, __fsub_rn(x, v[q]));
                        }
                        tmem_ld<8>(tbase + 8 * h + TC_N, rb);
                        tmem_ld<8>(tbase + 8 * h, ra);
                        tmem_wait<8>(rb);
                        tmem_wait<8>(ra);
                        if (h == 3) release(free_bar[1]);
#pragma unroll
                        for (int q = 0; q < 8; ++q)
                            add_chunk<6>(f(ra[q]), f(rb[q]), f(r2[8 * h + q]), v[q], ev[q], hi[8 * h + q], lo[8 * h + q]);
                    }
                    release(high_bar);
                } else {
                    // acc_0 and acc_1 first, then the rest 8 columns at a time
                    uint32_t r0[32], r1[32];
                    tmem_ld<32>(tbase, r0);
                    tmem_ld<32>(tbase + TC_N, r1);
                    tmem_wait<32>(r0);
                    tmem_wait<32>(r1);
                    release(free_bar[0]);
#pragma unroll
                    for (int h = 0; h < 4; ++h) {
                        uint32_t ra[8], rb[8], rc[8];
                        tmem_ld<8>(thigh + 8 * h + TC_N * 4, ra);
                        tmem_ld<8>(thigh + 8 * h + TC_N * 3, rb);
                        tmem_ld<8>(thigh + 8 * h + TC_N * 2, rc);
                        tmem_wait<8>(ra);
                        tmem_wait<8>(rb);
                        tmem_wait<8>(rc);
#pragma unroll
                        for (int q = 0; q < 8; ++q)
                            add_chunk<5>(f(r0[8 * h + q]), f(r1[8 * h + q]), f(rc[q]), __fmaf_rn(f(ra[q]), 0x1p-8f, f(rb[q])),
                                         0.f, hi[8 * h + q], lo[8 * h + q]);
                    }
                    release(high_bar);
                }
            }
            if (!ok) break;
            // results: exact conversions and the power-of-two scaling on the bit
            // patterns, one or two FP64 instructions per output
            const int i = it.i0 + 32 * quad + lane, jb = it.j0 + c0;
            const int ei = i < M ? ex[i] - 14 : 0;
            const int row4 = i & ~3, a = lane & 3;
#pragma unroll
            for (int g = 0; g < 4; ++g) {
                double2 p[4];
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    const int q = 8 * g + u, j = jb + q;
                    double l = f2d_normal(lo[q]);
                    if constexpr (SL == 7) l += f2d_normal(mid[q]);
                    const double x = scale2(f2d_normal(hi[q]) + l, ei + (j < N ? ey[j] : 0));
                    if (u & 1) p[u / 2].y = x;
                    else p[u / 2].x = x;
                    // the mirror image: consecutive rows of a column
                    if (w.lower && j < i && i < M) {
                        if (atomic) atomicAdd(&C[(size_t)j * ldc + i], x);
                        else C[(size_t)j * ldc + i] = x;
                    }
                }
                // 4 x 4 transpose of column pairs among four lanes: lane a gets
                // pair a of the four rows, so that a warp writes 64-byte pieces
#pragma unroll
                for (int b = 1; b <= 2; b <<= 1)
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        if (k & b) continue;
                        const bool up = (a & b) != 0;
                        const double2 send = up ? p[k] : p[k | b];
                        const double2 got = make_double2(__shfl_xor_sync(0xffffffffu, send.x, b),
                                                         __shfl_xor_sync(0xffffffffu, send.y, b));
                        if (up) p[k] = got;
                        else p[k | b] = got;
                    }
                const int j = jb + 8 * g + 2 * a;
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const int r = row4 + k;
                    if (r >= M || j >= N) continue;
                    double *cr = C + (size_t)r * ldc + j;
                    if (vec && j + 1 < N) {
                        *reinterpret_cast<double2 *>(cr) = p[k];
                        continue;
                    }
#pragma unroll
                    for (int u = 0; u < 2; ++u) {
                        if (j + u >= N || (w.lower && j + u > r)) continue;
                        const double x = u ? p[k].y : p[k].x;
                        if (atomic) atomicAdd(cr + u, x);
                        else cr[u] = x;
                    }
                }
            }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    if (warp == 1)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(TC_TMEM_COLS));
}

// ---- the product of the magnitudes ------------------------------------------
//
// h = X Y^T of one slice of magnitudes each (all terms positive, FP32
// accumulators: a lower bound to 2^-13), per 128 x 64 nt item (nt <= 4 blocks of 64
// columns, so that the first operand is read ntn / nt times) over a range of K.
// Four K steps to a stage (one wait and one commit per four MMAs), two sets of
// accumulators.  Either h is added to chk.h (ld N), or it is checked against the
// sums of the rows' and columns' magnitudes and the tiles that fail are marked.
// What bounds it: the loads.  Update of 163,842 x 300 x 300 (98 MB of magnitudes):
// 57 us; as one-block items with a stage per K step 205.  Roles, waits and
// teardown as k_ozaki_tc's.
constexpr int kMagSteps = 4, kMagBlocks = 4, kMagStages = 4;
constexpr uint32_t kMagA = 2u * TC_M * TC_K, kMagB = 2u * TC_N * TC_K;  // bytes per K step and block
constexpr uint32_t kMagStage = kMagSteps * (kMagA + kMagBlocks * kMagB);
constexpr size_t kMagSmem = (size_t)kMagStages * kMagStage + 1024;

struct MagWork {
    int groups, tiles, items;  // column groups, output tiles, tiles x K ranges
    int nt, nby;               // column blocks per group, of the second operand
    int ksteps, split;         // K steps of the product, K steps per item
};
struct MagCheck {
    float *h;
    const float *lx, *ly;  // limits; ly in whole blocks of 64 columns
    float ratio;
    int *tiles;
    int tiles_ld;
};

__global__ void __launch_bounds__(TC_THREADS, 1)
    k_magnitudes_tc(int M, int N, const __nv_bfloat16 *__restrict__ Xs, int nbx, const __nv_bfloat16 *__restrict__ Ys,
                    MagWork w, MagCheck chk, int *__restrict__ err) {
    extern __shared__ unsigned char smem_dyn[];
    __shared__ __align__(8) uint64_t full_bar[kMagStages], empty_bar[kMagStages], accf_bar[2], free_bar[2], drain_bar;
    __shared__ uint32_t tmem_slot;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t smem0 = (smem_addr(smem_dyn) + 1023u) & ~1023u;
    if (threadIdx.x == 0) {
        for (int st = 0; st < kMagStages; ++st) {
            mbar_init(smem_addr(&full_bar[st]), 1);
            mbar_init(smem_addr(&empty_bar[st]), 1);
        }
        for (int q = 0; q < 2; ++q) {
            mbar_init(smem_addr(&accf_bar[q]), 1);
            mbar_init(smem_addr(&free_bar[q]), TC_DRAIN_WARPS);
        }
        mbar_init(smem_addr(&drain_bar), 1);
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_addr(&tmem_slot)),
                     "r"(TC_TMEM_COLS));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n");
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    const uint32_t tmem = tmem_slot;
    // item -> row tile, first column block, blocks, first K step, K steps
    struct Item {
        int ti, jb, nb, kc0, nk;
    };
    auto item_of = [&](int item) {
        const int sp = item / w.tiles, tile = item - sp * w.tiles, ti = tile / w.groups;
        Item it;
        it.ti = ti;
        it.jb = (tile - ti * w.groups) * w.nt;
        it.nb = min(w.nt, w.nby - it.jb);
        it.kc0 = sp * w.split;
        it.nk = min(w.split, w.ksteps - it.kc0);
        return it;
    };
    if (warp == 0) {
        if (lane == 0) {
            bool ok = true;
            int g = 0;  // stages filled by this CTA so far
            for (int item = blockIdx.x; item < w.items && ok; item += gridDim.x) {
                const Item it = item_of(item);
                for (int k0 = 0; k0 < it.nk; k0 += kMagSteps, ++g) {
                    const int st = g % kMagStages, steps = min(kMagSteps, it.nk - k0);
                    if (g >= kMagStages) ok = mbar_wait(smem_addr(&empty_bar[st]), ((g / kMagStages) & 1) ^ 1, err);
                    if (!ok) break;
                    const uint32_t fb = smem_addr(&full_bar[st]), dst = smem0 + st * kMagStage;
                    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(fb),
                                 "r"(steps * (kMagA + it.nb * kMagB))
                                 : "memory");
                    for (int q = 0; q < steps; ++q) {
                        const size_t kc = it.kc0 + k0 + q;
                        bulk_load(dst + q * kMagA, Xs + (kc * nbx + it.ti) * (kMagA / 2), kMagA, fb);
                        bulk_load(dst + kMagSteps * kMagA + q * kMagBlocks * kMagB, Ys + (kc * w.nby + it.jb) * (kMagB / 2),
                                  it.nb * kMagB, fb);
                    }
                }
            }
            for (int q = max(0, g - kMagStages); q < g; ++q)
                mbar_wait(smem_addr(&full_bar[q % kMagStages]), (q / kMagStages) & 1, err);
        }
    } else if (warp == 1) {
        const uint32_t el = elect_lane();
        constexpr uint32_t LBO = 128, SBO = 256;
        bool ok = true;
        uint32_t g = 0, c = 0;  // stages and items so far
        for (int item = blockIdx.x; item < w.items && ok; item += gridDim.x, ++c) {
            const Item it = item_of(item);
            const uint32_t d = tmem + (c & 1) * TC_N * kMagBlocks, idesc = umma_idesc(TC_M, TC_N * it.nb);
            // the set is drained of the item before the last
            if (c >= 2) ok = mbar_wait(smem_addr(&free_bar[c & 1]), ((c >> 1) - 1) & 1, err);
            if (!ok) break;
            asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
            for (int k0 = 0; k0 < it.nk; k0 += kMagSteps, ++g) {
                const uint32_t st = g % kMagStages;
                ok = mbar_wait(smem_addr(&full_bar[st]), (g / kMagStages) & 1, err);
                if (!ok) break;
                const uint32_t a = smem0 + st * kMagStage, b = a + kMagSteps * kMagA;
                const int steps = min(kMagSteps, it.nk - k0);
                for (int q = 0; q < steps; ++q)
                    umma_f16(d, umma_desc(umma_desc_lo(a + q * kMagA, LBO), SBO),
                             umma_desc(umma_desc_lo(b + q * kMagBlocks * kMagB, LBO), SBO), idesc, k0 + q > 0, el);
                umma_commit(smem_addr(&empty_bar[st]), el);
            }
            if (!ok) break;
            umma_commit(smem_addr(&accf_bar[c & 1]), el);
        }
        umma_commit(smem_addr(&drain_bar), el);
        mbar_wait(smem_addr(&drain_bar), 0, err);
    } else {
        const int quad = warp & 3, c0 = 32 * ((warp - 2) >> 2);
        bool ok = true;
        int c = 0;
        for (int item = blockIdx.x; item < w.items && ok; item += gridDim.x, ++c) {
            const Item it = item_of(item);
            const int i = it.ti * TC_M + 32 * quad + lane;
            const float li = chk.h || i >= M ? 0.f : chk.lx[i];
            ok = __all_sync(0xffffffffu, mbar_wait(smem_addr(&accf_bar[c & 1]), (c >> 1) & 1, err));
            if (!ok) break;
            asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
            for (int b = 0; b < it.nb; ++b) {
                uint32_t r[32];
                tmem_ld<32>(tmem + ((uint32_t)(32 * quad) << 16) + (c & 1) * TC_N * kMagBlocks + b * TC_N + c0, r);
                tmem_wait<32>(r);
                if (b == it.nb - 1) {
                    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
                    __syncwarp();
                    if (lane == 0) mbar_arrive(smem_addr(&free_bar[c & 1]));
                }
                const int jb = (it.jb + b) * TC_N + c0;
                if (chk.h) {
                    if (i < M)
#pragma unroll
                        for (int q = 0; q < 32; ++q)
                            if (jb + q < N) atomicAdd(&chk.h[(size_t)i * N + jb + q], __uint_as_float(r[q]));
                    continue;
                }
                bool fails = false;
#pragma unroll
                for (int q = 0; q < 32; q += 4) {
                    const float4 l = *reinterpret_cast<const float4 *>(chk.ly + jb + q);
                    fails |= digits_fail(li, l.x, chk.ratio, __uint_as_float(r[q])) |
                             digits_fail(li, l.y, chk.ratio, __uint_as_float(r[q + 1])) |
                             digits_fail(li, l.z, chk.ratio, __uint_as_float(r[q + 2])) |
                             digits_fail(li, l.w, chk.ratio, __uint_as_float(r[q + 3]));
                }
                fails = fails && i < M;
                if (__any_sync(0xffffffffu, fails) && lane == 0)
                    chk.tiles[(size_t)((it.ti * TC_M + 32 * quad) >> 6) * chk.tiles_ld + it.jb + b] = 1;
            }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    if (warp == 1)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(TC_TMEM_COLS));
}

inline int round_up(int x, int m) { return (x + m - 1) / m * m; }
inline bool aligned16(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }
// rows of FP64 pairs can be read (written) as 16-byte vectors
inline bool pair_rows(const double *p, int ld) { return aligned16(p) && ld % 2 == 0; }

template <int SL>
void launch_tc(cudaStream_t s, const OzakiOperand &X, const OzakiOperand &Y, double *C, int ldc, const TcWork &w,
               bool atomic, int *err) {
    HSIM_SMEM_LIMIT_ONCE(k_ozaki_tc<SL>, tc_smem<SL>());
    const int grid = std::min(w.items, sm_count_oz());
    const bool vec = !atomic && !w.lower && pair_rows(C, ldc);
    k_ozaki_tc<SL><<<grid, TC_THREADS, tc_smem<SL>(), s>>>(X.rows, Y.rows, X.slices, X.rows_p / TC_M, Y.slices,
                                                          Y.rows_p / TC_N, X.exps, Y.exps, C, ldc, w, atomic ? 1 : 0,
                                                          vec ? 1 : 0, err);
    HSIM_LAUNCHED();
}

}  // namespace

// Scratch: digits x rows_p x kp BF16 digits then rows_p exponents, rounded to
// whole 512-byte blocks so operands placed back to back in one buffer stay
// aligned for the bulk copies (either operand's row padding).
static size_t operand_bytes(int rows, int kdim, int digits) {
    const size_t rows_p = (size_t)round_up(std::max(rows, 1), TC_M), kp = (size_t)round_up(std::max(kdim, 1), TC_K);
    size_t b = (size_t)digits * rows_p * kp * sizeof(__nv_bfloat16) + sizeof(int) * rows_p;
    return (b + 511) / 512 * 512;
}

size_t ozaki_cols_scratch(int n, int cols, int digits) { return operand_bytes(cols, n, digits); }
size_t ozaki_rows_scratch(int rows, int k, int digits) { return operand_bytes(rows, k, digits); }

static OzakiOperand make_operand(int rows, int kdim, void *scratch, int digits, OzakiRole role) {
    HSIM_CHECK_ARG(digits == 1 || (digits >= 5 && digits <= 7), "ozaki product: 5, 6 or 7 digits per value");
    HSIM_CHECK_ARG(aligned16(scratch), "ozaki product: scratch not 16-byte aligned");
    OzakiOperand op;
    op.digits = digits;
    op.role = role;
    op.rows = rows;
    op.rows_p = round_up(std::max(rows, 1), role == OzakiRole::X ? TC_M : TC_N);
    op.kp = round_up(std::max(kdim, 1), TC_K);
    op.slices = static_cast<__nv_bfloat16 *>(scratch);
    op.exps = reinterpret_cast<int *>(op.slices + (size_t)digits * op.rows_p * op.kp);
    return op;
}

static int role_log(OzakiRole r) { return r == OzakiRole::X ? 7 : 6; }

// exponents (preset: kNoExp) and, where they are asked for, sums (added) of one or
// two blocks of n rows
static void launch_col_exps(cudaStream_t s, int n, const ExpsArgs &a, const ExpsArgs *b, const int *rexp) {
    // rows per CTA: about eight CTAs per SM, 32 to 1024 rows
    const int64_t ca = cdiv(a.C, 64), cb = b ? cdiv(b->C, 64) : 0;
    const int64_t want = std::max<int64_t>(1, 8 * (int64_t)sm_count_oz() / (ca + cb));
    const int rows = (int)std::min<int64_t>(1024, std::max<int64_t>(32, round_up((int)cdiv(n, want), 8)));
    const dim3 g(cdiv(n, rows), (unsigned)std::max(ca, cb), b ? 2 : 1);
    auto go = [&](auto kernel) { kernel<<<g, 256, 0, s>>>(n, a, b ? *b : a, rows, rexp); };
    if (rexp) go(k_col_exps<true, false>);
    else if (a.sums) go(k_col_exps<false, true>);
    else go(k_col_exps<false, false>);
    HSIM_LAUNCHED();
}

static void ozaki_col_exps(cudaStream_t s, int n, int cols, const double *X, int ldx, int *exps, const int *rexp,
                           double *sums = nullptr) {
    k_fill_int<<<cdiv(cols, 256), 256, 0, s>>>(cols, kNoExp, exps);
    HSIM_LAUNCHED();
    launch_col_exps(s, n, {X, cols, ldx, pair_rows(X, ldx), exps, sums}, nullptr, rexp);
}

// n rows of X (and of X2 into op2, of the same K and digits)
static void split_cols_into(cudaStream_t s, const OzakiOperand &op, int n, const double *X, int ldx, const int *rexp,
                            float *sums = nullptr, const OzakiOperand *op2 = nullptr, const double *X2 = nullptr,
                            int ldx2 = 0) {
    auto args = [](const OzakiOperand &o, const double *x, int ld) {
        return SplitArgs{x, o.rows, ld, pair_rows(x, ld), o.exps, o.slices, o.rows_p, role_log(o.role)};
    };
    const SplitArgs a = args(op, X, ldx), b = op2 ? args(*op2, X2, ldx2) : a;
    // four blocks per SM (shared memory), each with up to eight tiles
    const int nt = cdiv(op.kp, 32), ca = cdiv(a.rows_p, 64), cb = op2 ? cdiv(b.rows_p, 64) : 0;
    const int tiles =
        (int)std::max<int64_t>(1, std::min<int64_t>(8, (int64_t)nt * (ca + cb) / (4 * (int64_t)sm_count_oz())));
    const dim3 g(cdiv(nt, tiles), std::max(ca, cb), op2 ? 2 : 1);
    auto go = [&](auto kernel) {
        kernel<<<g, 256, kSplitSmem, s>>>(n, a, b, rexp, op.kp, sums, tiles);
        HSIM_LAUNCHED();
    };
    if (op.digits == 5) {
        HSIM_SMEM_LIMIT_ONCE(k_split_cols<5>, kSplitSmem);
        go(k_split_cols<5>);
    } else if (op.digits == 6) {
        HSIM_SMEM_LIMIT_ONCE(k_split_cols<6>, kSplitSmem);
        go(k_split_cols<6>);
    } else if (op.digits == 1) {
        HSIM_SMEM_LIMIT_ONCE(k_split_cols<1>, kSplitSmem);
        go(k_split_cols<1>);
    } else {
        HSIM_SMEM_LIMIT_ONCE(k_split_cols<7>, kSplitSmem);
        go(k_split_cols<7>);
    }
}

OzakiOperand ozaki_split_cols(cudaStream_t s, int n, int cols, const double *X, int ldx, void *scratch, int digits,
                              OzakiRole role) {
    OzakiOperand op = make_operand(cols, n, scratch, digits, role);
    if (n <= 0 || cols <= 0) return op;
    ozaki_col_exps(s, n, cols, X, ldx, op.exps, nullptr);
    split_cols_into(s, op, n, X, ldx, nullptr);
    return op;
}

// mags, limits (may be null): the magnitudes' slice and limits of every row as well
static void split_rows_into(cudaStream_t s, const OzakiOperand &op, int k, const double *X, int ldx, const int *cexp,
                            __nv_bfloat16 *mags = nullptr, float *limits = nullptr) {
    k_row_exps<<<cdiv(op.rows, 8), 256, 0, s>>>(op.rows, k, X, ldx, cexp, op.exps, limits);
    HSIM_LAUNCHED();
    const unsigned g = cdiv((int64_t)(op.rows_p / 8) * ((op.kp + 31) / 32) * 32, 256);
    const bool vec = pair_rows(X, ldx);
    const int rl = role_log(op.role);
    auto go = [&](auto kernel) {
        kernel<<<g, 256, 0, s>>>(op.rows, k, X, ldx, vec, op.exps, cexp, op.slices, op.rows_p, op.kp, rl, mags);
        HSIM_LAUNCHED();
    };
    if (op.digits == 5) go(k_split_rows<5>);
    else if (op.digits == 6) go(k_split_rows<6>);
    else go(k_split_rows<7>);
}

OzakiOperand ozaki_split_rows(cudaStream_t s, int rows, int k, const double *X, int ldx, void *scratch, int digits) {
    OzakiOperand op = make_operand(rows, k, scratch, digits, OzakiRole::X);
    if (rows <= 0) return op;
    split_rows_into(s, op, k, X, ldx, nullptr);
    return op;
}

// work items of C = X Y^T; splits <= 0 chooses the number of K ranges, which is
// returned
static int plan_tc(const OzakiOperand &X, const OzakiOperand &Y, int splits, bool lower, TcWork &w) {
    HSIM_CHECK_ARG(X.kp == Y.kp, "ozaki_product: operands split over different K");
    HSIM_CHECK_ARG(X.digits == Y.digits, "ozaki_product: operands split into different digit counts");
    HSIM_CHECK_ARG(X.role == OzakiRole::X && Y.role == OzakiRole::Y, "ozaki_product: operand roles");
    HSIM_CHECK_ARG(!lower || X.rows == Y.rows, "ozaki product: lower triangle needs a square result");
    w.lower = lower ? 1 : 0;
    w.ksteps = X.kp / TC_K;
    w.ntn = (int)cdiv(Y.rows, TC_N);
    const int tx = (int)cdiv(X.rows, TC_M);
    int64_t tiles = 0;
    for (int r = 0; r < tx; ++r) tiles += lower ? std::min(w.ntn, 2 * r + 2) : w.ntn;
    // K ranges: whole chunks, at most kItemK rows each, chosen so that tiles x
    // ranges fill whole waves of one CTA per SM
    const int64_t chunks = cdiv(w.ksteps, kChunkSteps);
    const int64_t s_min = std::max<int64_t>(1, cdiv((int64_t)w.ksteps * TC_K, kItemK));
    if (splits <= 0) {
        const int64_t sms = sm_count_oz();
        const int64_t s_max = std::max(s_min, std::min<int64_t>(chunks, 8 * sms / tiles + 1));
        double best = -1.0;
        for (int64_t sp = s_min; sp <= s_max; ++sp) {
            const int64_t items = tiles * sp, waves = (items + sms - 1) / sms;
            // fill of the last wave, with a small preference for fewer ranges
            const double eff = (double)items / (double)(waves * sms) - 0.002 * (double)sp;
            if (eff > best + 1e-9) {
                best = eff;
                splits = (int)sp;
            }
        }
    }
    splits = (int)std::max<int64_t>(splits, s_min);
    w.split = (int)cdiv(chunks, splits) * kChunkSteps;
    splits = (int)cdiv(w.ksteps, w.split);
    HSIM_CHECK_ARG(tiles * splits <= INT32_MAX / 2, "ozaki product: too many tiles");
    w.tiles = (int)tiles;
    w.items = (int)(tiles * splits);
    return splits;
}

static void zero_block(cudaStream_t s, int rows, int cols, double *C, int ldc) {
    if (ldc == cols) HSIM_CUDA(cudaMemsetAsync(C, 0, (size_t)rows * cols * sizeof(double), s));
    else HSIM_CUDA(cudaMemset2DAsync(C, (size_t)ldc * sizeof(double), 0, (size_t)cols * sizeof(double), rows, s));
}

void ozaki_product(cudaStream_t s, const OzakiOperand &X, const OzakiOperand &Y, double *C, int ldc, int splits, int *err,
                   bool lower, bool accumulate, const int *skip, int skip_ld) {
    if (X.rows <= 0 || Y.rows <= 0) return;
    TcWork w{};
    splits = plan_tc(X, Y, splits, lower, w);
    w.skip = skip;
    w.skip_ld = skip_ld;
    const bool atomic = splits > 1 || accumulate;
    if (atomic && !accumulate) zero_block(s, X.rows, Y.rows, C, ldc);
    if (X.digits == 5) launch_tc<5>(s, X, Y, C, ldc, w, atomic, err);
    else if (X.digits == 6) launch_tc<6>(s, X, Y, C, ldc, w, atomic, err);
    else launch_tc<7>(s, X, Y, C, ldc, w, atomic, err);
}

// the product of two slices of magnitudes, added to chk.h (over K ranges that fill
// the SMs) or checked (one K range)
static void product_magnitudes(cudaStream_t s, const OzakiOperand &X, const OzakiOperand &Y, const MagCheck &chk, int *err) {
    MagWork w{};
    w.nby = Y.rows_p / TC_N;
    w.groups = (int)cdiv(w.nby, kMagBlocks);
    w.nt = (int)cdiv(w.nby, w.groups);
    w.ksteps = X.kp / TC_K;
    const int64_t tiles = (int64_t)(X.rows_p / TC_M) * w.groups;
    const int64_t want = chk.h ? std::max<int64_t>(1, (int64_t)sm_count_oz() / tiles) : 1;
    const int64_t stages = cdiv(w.ksteps, kMagSteps);
    w.split = (int)(kMagSteps * cdiv(stages, std::min(stages, want)));
    const int64_t items = tiles * cdiv(w.ksteps, w.split);
    HSIM_CHECK_ARG(items <= INT32_MAX / 2, "ozaki product: too many tiles");
    w.tiles = (int)tiles;
    w.items = (int)items;
    HSIM_SMEM_LIMIT_ONCE(k_magnitudes_tc, kMagSmem);
    k_magnitudes_tc<<<std::min(w.items, sm_count_oz()), TC_THREADS, kMagSmem, s>>>(X.rows, Y.rows, X.slices, X.rows_p / TC_M,
                                                                              Y.slices, w, chk, err);
    HSIM_LAUNCHED();
}

// ---- products over ranges of rows -------------------------------------------
// The digits of a whole n x 750 block are 5 to 7 n x 1.5 KB (2.3 GB at 250,000
// rows and six digits); a range of rows keeps the scratch near kRangeBytes at
// any n.  Ranges are whole work items of the product (kItemK rows for a Gram,
// which adds the ranges in FP64 as it adds its items).
constexpr size_t kRangeBytes = (size_t)1 << 30;

static int range_rows(int64_t n, size_t row_bytes, int unit) {
    const int64_t most = std::max<int64_t>(unit, (int64_t)(kRangeBytes / row_bytes) / unit * unit);
    const int64_t ranges = std::max<int64_t>(1, (n + most - 1) / most);
    return (int)std::min<int64_t>(most, ((n + ranges - 1) / ranges + unit - 1) / unit * unit);
}
static size_t exps_bytes(int rows) { return ((size_t)rows * sizeof(int) + 511) / 512 * 512; }
static int gram_rows(int n, int ka, int kb, int digits) {
    return range_rows(n, 2 * (size_t)digits * (round_up(ka, TC_M) + round_up(kb, TC_N)), kItemK);
}

size_t ozaki_gram_scratch(int n, int ka, int kb, int digits) {
    const int r = std::min(gram_rows(n, ka, kb, digits), n);
    return exps_bytes(ka) + exps_bytes(kb) + operand_bytes(ka, r, digits) + operand_bytes(kb, r, digits);
}

void ozaki_gram(cudaStream_t s, int n, int ka, int kb, const double *A, int lda, const double *B, int ldb, double *G,
                int ldg, int digits, void *scratch, int *err) {
    const int range = gram_rows(n, ka, kb, digits);
    int *ex = static_cast<int *>(scratch);
    int *ey = ex + exps_bytes(ka) / sizeof(int);
    unsigned char *sx = reinterpret_cast<unsigned char *>(ey) + exps_bytes(kb);
    unsigned char *sy = sx + operand_bytes(ka, std::min(range, n), digits);
    k_fill_int<<<cdiv((ey - ex) + kb, 256), 256, 0, s>>>((int)(ey - ex) + kb, kNoExp, ex);
    HSIM_LAUNCHED();
    const ExpsArgs ea{A, ka, lda, pair_rows(A, lda), ex, nullptr}, eb{B, kb, ldb, pair_rows(B, ldb), ey, nullptr};
    launch_col_exps(s, n, ea, &eb, nullptr);
    const bool several = n > range;
    if (several) HSIM_CUDA(cudaMemset2DAsync(G, (size_t)ldg * sizeof(double), 0, (size_t)kb * sizeof(double), ka, s));
    for (int r0 = 0; r0 < n; r0 += range) {
        const int rows = std::min(range, n - r0);
        OzakiOperand X = make_operand(ka, rows, sx, digits, OzakiRole::X), Y = make_operand(kb, rows, sy, digits, OzakiRole::Y);
        X.exps = ex;
        Y.exps = ey;
        split_cols_into(s, X, rows, A + (size_t)r0 * lda, lda, nullptr, nullptr, &Y, B + (size_t)r0 * ldb, ldb);
        ozaki_product(s, X, Y, G, ldg, 0, err, false, several);
    }
}

static int update_rows(int n, int k, int digits) { return range_rows(n, 2 * (size_t)digits * round_up(k, TC_K), TC_M); }

size_t ozaki_update_scratch(int n, int k, int m, int digits) {
    return operand_bytes(m, k, digits) + operand_bytes(std::min(update_rows(n, k, digits), n), k, digits);
}

void ozaki_update(cudaStream_t s, int n, int k, int m, const double *A, int lda, const double *B, int ldb, double *C,
                  int ldc, int digits, void *scratch, int *err) {
    const int range = update_rows(n, k, digits);
    unsigned char *sy = static_cast<unsigned char *>(scratch), *sx = sy + operand_bytes(m, k, digits);
    OzakiOperand Y = ozaki_split_cols(s, k, m, B, ldb, sy, digits, OzakiRole::Y);
    for (int r0 = 0; r0 < n; r0 += range) {
        OzakiOperand X = ozaki_split_rows(s, std::min(range, n - r0), k, A + (size_t)r0 * lda, lda, sx, digits);
        ozaki_product(s, X, Y, C + (size_t)r0 * ldc, ldc, 1, err);
    }
}

// ---- FP64 products on seven digits --------------------------------------------
// gram and gemm_nn of the FP64 path.  Seven digits keep 55 bits against each
// group's maximum and the digit pairs down to 2^-63, so the error per term is
// 2^-56 of max|x| max|y| where an FP64 accumulation rounds every partial sum to
// 2^-54 of itself.  Against quad-precision sums, FP64 kernels and digits:
// Gram of 163,842 x 300 5.3e-16 and 0.9e-16 (all positive 4.7 and 1.4, smooth
// columns 23 and 1.6), update 5.8e-16 and 2.3e-16 (a random second factor 5.8 and
// 0.6, columns scaled by 10^+-6 5.7 and 2.2); the same order at 5,003 to 20,011
// rows and 77 to 750 columns.  Tiles where the maxima say too little go to the
// FP64 kernels (digits_fail and k_guard_tiles above), which the device decides
// before a digit of them is multiplied.  A Gram's columns have their own
// exponents; an update scales column k of A by 2^-c_k and row k of B by 2^c_k,
// exactly, so that their mean magnitudes meet (means: one large entry must not move
// the scale of the others).
//
// What the check costs (calls with a wait, without and with it): Gram 163,842 x 300
// 1,407 and 1,445 us, 1,024 x 300 110 and 120; update 163,842 x 300 1,124 and 1,172,
// 1,024 x 165 97 and 111.  Inputs that it sends to the FP64 kernel pay for it there:
// a Gram of 16,384 x 75 530 -> 670, of 163,842 x 300 28,000 to 33,000 with every row
// of tiles flagged, 14,900 with one column.
//
// Where the line lies (us, FP64 kernel / digits, calls with a wait): Gram 1,024
// rows x 30 to 300 columns 281 / 100 to 283 / 120, 16,384 x 75 530 / 139, 163,842 x
// 300 33,000 / 1,445; fewer rows than 1,024 are left to the FP64 kernel (its time
// falls with them, and the rule on standing-out entries has no room).  Update
// with k = 30 44 / 57 to 8,192 rows and 75 / 60 at 16,384, k = 50 77 / 55 from
// 1,024 rows on (the solve's form, without the check), 163,842 x 300 25,700 / 1,172.
// A context's first call also
// allocates the scratch, about 140 us: where the scratch is not held by the caller
// an update takes the digits only if the FP64 kernel is slower than both (about 1.5
// us per inner term when it waits for its chain, 1.1 TFLOP/s otherwise; 15,923 x 36
// 130 us against 97, but 237 in a first call).
constexpr int kDigits64 = 7;
constexpr int kUpdate64MaxK = 4096;  // the inner sums of the measurements above

bool gram64_on_digits(int n, int ka, int kb) { return n >= 1024 && (double)n * ka * kb >= 5e5; }
bool update64_on_digits(int n, int k, int m, bool held) {
    const double work = (double)n * k * m;
    if (k > kUpdate64MaxK) return false;
    return held ? (k > 40 && work >= 2e6) || work >= 1.2e7 : (k >= 165 && work >= 2e6) || work >= 1.2e8;
}

namespace {

// Powers of two c_k: half the gap between the mean magnitudes of column k of A (sum
// over n rows) and row k of B (sum in units of 2^eb over m columns), less the mean
// gap of all k (a common factor does nothing); below 1.5 left at 0, so that pairs
// alike are not told apart by rounding.  One CTA; zeros and infinities: 0.  ey (m):
// preset for k_col_exps.
__global__ void __launch_bounds__(256) k_balance(int k, int n, int m, const double *__restrict__ suma,
                                                 const int *__restrict__ eb, const float *__restrict__ sumb,
                                                 int *__restrict__ c, int *__restrict__ ey) {
    __shared__ float red[2][8];
    for (int j = threadIdx.x; j < m; j += 256) ey[j] = kNoExp;
    auto log2_of = [](double x, float &l) {
        const int h = __double2hiint(x), e = (h >> 20) & 0x7FF;
        l = (float)(e - 1023) + __log2f(__int_as_float(0x3F800000 | ((h & 0xFFFFF) << 3)));
        return e != 0 && e != 0x7FF;
    };
    auto gap = [&](int j, float &g) {
        float a, b;
        const bool ok = log2_of(suma[j], a) && log2_of((double)sumb[j], b) && !bad_exp(eb[j]);
        g = 0.5f * ((a - __log2f((float)n)) - (b + (float)eb[j] - __log2f((float)m)));
        return ok;
    };
    float sum = 0.f, cnt = 0.f, g;
    for (int j = threadIdx.x; j < k; j += 256)
        if (gap(j, g)) sum += g, cnt += 1.f;
    for (int o = 16; o > 0; o >>= 1) {
        sum += __shfl_xor_sync(0xffffffffu, sum, o);
        cnt += __shfl_xor_sync(0xffffffffu, cnt, o);
    }
    if ((threadIdx.x & 31) == 0) red[0][threadIdx.x >> 5] = sum, red[1][threadIdx.x >> 5] = cnt;
    __syncthreads();
    sum = cnt = 0.f;
    for (int q = 0; q < 8; ++q) sum += red[0][q], cnt += red[1][q];
    const float mean = sum / fmaxf(cnt, 1.f);
    for (int j = threadIdx.x; j < k; j += 256) c[j] = gap(j, g) && fabsf(g - mean) > 1.5f ? __float2int_rn(g - mean) : 0;
}

// 512-byte aligned pieces of one scratch block
struct Pieces {
    unsigned char *p;
    size_t used = 0;
    template <class T> T *take(size_t count) {
        T *q = reinterpret_cast<T *>(p + used);
        used += (count * sizeof(T) + 511) / 512 * 512;
        return q;
    }
};

// 64 x 64 tiles of an M x N result (whole row tiles of the products)
inline int tile_rows(int M) { return 2 * (int)cdiv(M, TC_M); }
inline int tile_cols(int N) { return (int)cdiv(N, TC_N); }

// every how manieth row stands for all: 8 where that leaves 2048 and more, 4 below
// (a row pitch that an int holds)
int sample_step(int n, int ld) { return ld > INT32_MAX / 8 ? 1 : n >= 16384 ? 8 : 4; }

struct Gram64 {
    int range, step, sampled, mag_range;  // rows of a digit range; rows between sampled ones, their number, their range
    int *tiles, *ex, *ey;
    double *sx, *sy;
    float *h;
    unsigned char *dx, *dy;
    size_t zero_bytes, bytes;  // tiles to h; all of it
    Gram64(int n, int ka, int kb, int lda, int ldb, void *scratch) {
        Pieces q{static_cast<unsigned char *>(scratch)};
        range = std::min(gram_rows(n, ka, kb, kDigits64), n);
        step = sample_step(n, std::max(lda, ldb));
        sampled = (int)cdiv(n, step);
        mag_range = std::min(gram_rows(sampled, ka, kb, 1), sampled);
        tiles = q.take<int>((size_t)tile_rows(ka) * tile_cols(kb));
        sx = q.take<double>(ka);
        sy = q.take<double>(kb);
        h = q.take<float>((size_t)ka * kb);
        zero_bytes = q.used;
        ex = q.take<int>(ka);
        ey = q.take<int>(kb);
        dx = q.take<unsigned char>(std::max(operand_bytes(ka, range, kDigits64), operand_bytes(ka, mag_range, 1)));
        dy = q.take<unsigned char>(std::max(operand_bytes(kb, range, kDigits64), operand_bytes(kb, mag_range, 1)));
        bytes = q.used;
    }
};

struct Update64 {
    int range;
    int *tiles, *cexp, *bexp;
    double *suma;
    float *sumb, *lx, *ly;
    unsigned char *dy, *my, *dx, *mx;
    size_t zero_bytes, bytes;  // tiles to ly; all of it
    Update64(int n, int k, int m, void *scratch) {
        Pieces q{static_cast<unsigned char *>(scratch)};
        range = std::min(range_rows(n, 2 * (size_t)(kDigits64 + 1) * round_up(k, TC_K), TC_M), n);
        tiles = q.take<int>((size_t)tile_rows(n) * tile_cols(m));
        suma = q.take<double>(k);
        ly = q.take<float>(round_up(m, TC_N));
        zero_bytes = q.used;
        cexp = q.take<int>(k);
        bexp = q.take<int>(k);
        sumb = q.take<float>(k);
        lx = q.take<float>(range);
        dy = q.take<unsigned char>(operand_bytes(m, k, kDigits64));
        my = q.take<unsigned char>(operand_bytes(m, k, 1));
        dx = q.take<unsigned char>(operand_bytes(range, k, kDigits64));
        mx = q.take<unsigned char>(operand_bytes(range, k, 1));
        bytes = q.used;
    }
};

}  // namespace

size_t gram64_scratch(int n, int ka, int kb) { return Gram64(n, ka, kb, ka, kb, nullptr).bytes; }

void gram64(cudaStream_t s, int n, int ka, int kb, const double *A, int lda, const double *B, int ldb, double *G,
            int ldg, bool lower, Held held, void *scratch, int *err) {
    const Gram64 g(n, ka, kb, lda, ldb, scratch);
    const int tm = tile_rows(ka), tn = tile_cols(kb);
    HSIM_CUDA(cudaMemsetAsync(g.tiles, 0, g.zero_bytes, s));
    const bool same = A == B && ka == kb && lda == ldb;
    k_fill_int<<<cdiv((g.ey - g.ex) + kb, 256), 256, 0, s>>>((int)(g.ey - g.ex) + kb, kNoExp, g.ex);
    HSIM_LAUNCHED();
    const ExpsArgs ea{A, ka, lda, pair_rows(A, lda), g.ex, g.sx}, eb{B, kb, ldb, pair_rows(B, ldb), g.ey, g.sy};
    launch_col_exps(s, n, ea, same ? nullptr : &eb, nullptr);
    if (same) {
        HSIM_CUDA(cudaMemcpyAsync(g.ey, g.ex, (size_t)ka * sizeof(int), cudaMemcpyDeviceToDevice, s));
        HSIM_CUDA(cudaMemcpyAsync(g.sy, g.sx, (size_t)ka * sizeof(double), cudaMemcpyDeviceToDevice, s));
    }
    auto operands = [&](int rows, int digits, OzakiOperand &X, OzakiOperand &Y, const double *a, int la, const double *b,
                        int lb) {
        X = make_operand(ka, rows, g.dx, digits, OzakiRole::X);
        Y = make_operand(kb, rows, g.dy, digits, OzakiRole::Y);
        X.exps = g.ex;
        Y.exps = g.ey;
        split_cols_into(s, X, rows, a, la, nullptr, nullptr, &Y, b, lb);
    };
    OzakiOperand X, Y;
    if (held == Held::Entries) {
        MagCheck chk{};
        chk.h = g.h;
        for (int r0 = 0; r0 < g.sampled; r0 += g.mag_range) {
            const size_t r = (size_t)r0 * g.step;
            operands(std::min(g.mag_range, g.sampled - r0), 1, X, Y, A + r * lda, lda * g.step, B + r * ldb, ldb * g.step);
            product_magnitudes(s, X, Y, chk, err);
        }
        k_check_tiles<<<cdiv((int64_t)ka * kb, 256), 256, 0, s>>>(ka, kb, (float)n, digits_ratio(n), g.h, g.ex, g.sx, g.ey,
                                                                 g.sy, g.tiles, tn);
    } else {
        k_guard_tiles<<<dim3(tm, tn), 128, 0, s>>>(ka, kb, (double)n, g.ex, g.sx, g.ey, g.sy, g.tiles, tn);
    }
    HSIM_LAUNCHED();
    const bool several = n > g.range;
    if (several) zero_block(s, ka, kb, G, ldg);
    for (int r0 = 0; r0 < n; r0 += g.range) {
        operands(std::min(g.range, n - r0), kDigits64, X, Y, A + (size_t)r0 * lda, lda, B + (size_t)r0 * ldb, ldb);
        ozaki_product(s, X, Y, G, ldg, 0, err, lower, several, g.tiles, tn);
    }
    gram_tiles(s, n, ka, kb, A, lda, B, ldb, G, ldg, lower, g.tiles, tn);
}

size_t update64_scratch(int n, int k, int m) { return Update64(n, k, m, nullptr).bytes; }

void update64(cudaStream_t s, int n, int k, int m, const double *A, int lda, const double *B, int ldb, double *C,
              int ldc, Held held, void *scratch, int *err) {
    const Update64 u(n, k, m, scratch);
    const int tn = tile_cols(m);
    HSIM_CUDA(cudaMemsetAsync(u.tiles, 0, u.zero_bytes, s));
    // means over part of the rows: they only set the scale (the maxima beside them, in
    // cexp, are not used)
    const int step = sample_step(n, lda), sampled = (int)cdiv(n, step);
    launch_col_exps(s, sampled, {A, k, lda * step, pair_rows(A, lda * step), u.cexp, u.suma}, nullptr, nullptr);
    k_row_exps<<<cdiv(k, 8), 256, 0, s>>>(k, m, B, ldb, nullptr, u.bexp, u.sumb);
    HSIM_LAUNCHED();
    OzakiOperand Y = make_operand(m, k, u.dy, kDigits64, OzakiRole::Y), Ym = make_operand(m, k, u.my, 1, OzakiRole::Y);
    k_balance<<<1, 256, 0, s>>>(k, sampled, m, u.suma, u.bexp, u.sumb, u.cexp, Y.exps);
    HSIM_LAUNCHED();
    launch_col_exps(s, k, {B, m, ldb, pair_rows(B, ldb), Y.exps, nullptr}, nullptr, u.cexp);
    split_cols_into(s, Y, k, B, ldb, u.cexp);
    Ym.exps = Y.exps;
    const bool entries = held == Held::Entries;
    if (entries) {
        split_cols_into(s, Ym, k, B, ldb, u.cexp, u.ly);
        k_col_limits<<<cdiv(round_up(m, TC_N), 256), 256, 0, s>>>(m, round_up(m, TC_N), (float)k, Y.exps, u.ly);
        HSIM_LAUNCHED();
    }
    for (int r0 = 0; r0 < n; r0 += u.range) {
        const int rows = std::min(u.range, n - r0);
        int *tiles = u.tiles + (size_t)(r0 / 64) * tn;
        OzakiOperand X = make_operand(rows, k, u.dx, kDigits64, OzakiRole::X), Xm = make_operand(rows, k, u.mx, 1, OzakiRole::X);
        Xm.exps = X.exps;
        split_rows_into(s, X, k, A + (size_t)r0 * lda, lda, u.cexp, entries ? Xm.slices : nullptr, entries ? u.lx : nullptr);
        if (entries) {
            const MagCheck chk{nullptr, u.lx, u.ly, digits_ratio(k), tiles, tn};
            product_magnitudes(s, Xm, Ym, chk, err);
        } else {
            k_guard_tiles<<<dim3(cdiv(rows, 64), tn), 128, 0, s>>>(rows, m, (double)k, X.exps, nullptr, Y.exps, nullptr, tiles,
                                                                  tn);
            HSIM_LAUNCHED();
        }
        ozaki_product(s, X, Y, C + (size_t)r0 * ldc, ldc, 1, err, false, false, tiles, tn);
    }
    gemm_nn_tiles(s, n, k, m, A, lda, B, ldb, C, ldc, u.tiles, tn);
}

void ozaki_check(cudaStream_t s, int *err) {
    int h = 0;
    HSIM_CUDA(cudaMemcpyAsync(&h, err, sizeof(int), cudaMemcpyDeviceToHost, s));
    HSIM_CUDA(cudaStreamSynchronize(s));
    if (h != 0) {
        HSIM_CUDA(cudaMemsetAsync(err, 0, sizeof(int), s));
        HSIM_CUDA(cudaStreamSynchronize(s));
        fail(HSIM_E_INTERNAL, "tensor-core product: an mbarrier wait timed out");
    }
}

}  // namespace k
}  // namespace hsim
