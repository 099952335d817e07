// Dense symmetric eigensolver (FP64) for the Rayleigh-Ritz problems of Alg. 1
// and the coarsest-level problem of Alg. 3: the lowest m eigenpairs of a
// symmetric n x n matrix A.
//
//   1. Householder tridiagonalisation Q^T A Q = T in one cooperative launch:
//      per column k every CTA rebuilds the reflector v_k = (1, x_2..)/(x_1 -
//      beta) from the column below the diagonal (so no barrier is needed to
//      share it), computes p = tau A22 v over its rows of the trailing block,
//      forms w = p - (tau/2)(p.v) v and applies A22 -= v w^T + w v^T to its
//      rows.  Where the matrix fits in the CTAs' shared memory (n up to about
//      1650 on 152 SMs) each CTA keeps its rows there and one grid barrier per
//      column suffices (k_tridiag_rows, which takes the product with the column
//      before the reflector is known); otherwise the rows stay in global
//      memory with two barriers per column (k_tridiag).  The reflectors are
//      kept row-wise in Vh (contiguous for the back transformation).
//   2. Eigenvalues of T by multisection on division-free Sturm counts, a group
//      of lanes per index (ascending by construction): FP32 rounds, then FP64
//      rounds around the zero of the determinant's chord.
//   3. Eigenvectors of T: a column of the adjugate of T - lambda I from the two
//      Sturm sequences (k_tri_minors, k_tri_vectors).  Eigenvalues closer than
//      1e-9 ||T|| form a cluster, whose vectors come from inverse iteration
//      (Gaussian elimination with partial pivoting, reciprocal pivots kept),
//      three iterations from a hashed random start, made orthogonal to the
//      previous ones of the cluster in every iteration (one warp per cluster).
//   4. Back transformation X = Q Z: eight reflectors at a time in compact WY
//      form, a few eigenvectors per CTA held in registers (n <= 2048), else one
//      reflector at a time, the eigenvectors in shared memory.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cfloat>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <vector>

#include "common.h"
#include "kernels.h"

namespace cg = cooperative_groups;

namespace hsim {
namespace k {

namespace {

inline unsigned cdiv(int64_t a, int64_t b) { return (unsigned)((a + b - 1) / b); }

constexpr int kTriThreads = 256;
constexpr double kClusterTol = 1e-9;  // relative to ||T||
constexpr double kNearTol = 1e-4;     // the same, vectors made orthogonal once
constexpr size_t kTriSmemMax = 200 * 1024;  // dynamic shared memory limit of k_tridiag and k_tri_back

// sum over the block (256 threads); `red` holds 8 doubles; result in all threads
__device__ __forceinline__ double block_sum(double v, double *red) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    const int w = threadIdx.x >> 5;
    __syncthreads();  // red may still be read from the previous call
    if ((threadIdx.x & 31) == 0) red[w] = v;
    __syncthreads();
    double s = 0.0;
#pragma unroll
    for (int i = 0; i < kTriThreads / 32; ++i) s += red[i];
    return s;
}

__global__ void __launch_bounds__(kTriThreads) k_tridiag(int n, double *__restrict__ A, double *__restrict__ d,
                                                       double *__restrict__ e, double *__restrict__ tau,
                                                       double *__restrict__ Vh, double *__restrict__ p) {
    cg::grid_group grid = cg::this_grid();
    extern __shared__ double sm[];
    double *v = sm;       // n
    double *w = sm + n;   // n
    __shared__ double red[kTriThreads / 32];
    const int tid = threadIdx.x, lane = tid & 31;
    const int gwarp = (blockIdx.x * kTriThreads + tid) >> 5, nwarps = gridDim.x * (kTriThreads / 32);
    for (int k = 0; k + 1 < n; ++k) {
        const int L = n - k - 1;
        const double *col = A + (size_t)(k + 1) * n + k;  // x_i = col[i * n]
        double part = 0.0;
        for (int i = 1 + tid; i < L; i += kTriThreads) {
            const double x = col[(size_t)i * n];
            part += x * x;
        }
        const double sigma = block_sum(part, red);
        const double x0 = col[0];
        double beta = x0, t = 0.0, scale = 0.0;
        if (sigma != 0.0) {
            const double mu = sqrt(x0 * x0 + sigma);
            beta = x0 >= 0.0 ? -mu : mu;
            t = (beta - x0) / beta;
            scale = 1.0 / (x0 - beta);
        }
        for (int i = tid; i < L; i += kTriThreads) v[i] = i == 0 ? 1.0 : (t != 0.0 ? col[(size_t)i * n] * scale : 0.0);
        __syncthreads();
        if (blockIdx.x == 0) {
            if (tid == 0) {
                d[k] = A[(size_t)k * n + k];
                e[k] = beta;
                tau[k] = t;
            }
            for (int i = tid; i < L; i += kTriThreads) Vh[(size_t)k * n + k + 1 + i] = v[i];
        }
        if (t != 0.0) {
            // p = t A22 v, one warp per row
            for (int r = gwarp; r < L; r += nwarps) {
                const double *row = A + (size_t)(k + 1 + r) * n + k + 1;
                double s = 0.0;
                for (int j = lane; j < L; j += 32) s += row[j] * v[j];
                for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
                if (lane == 0) p[r] = t * s;
            }
            grid.sync();
            double pv = 0.0;
            for (int i = tid; i < L; i += kTriThreads) pv += p[i] * v[i];
            const double K = 0.5 * t * block_sum(pv, red);
            for (int i = tid; i < L; i += kTriThreads) w[i] = p[i] - K * v[i];
            __syncthreads();
            // A22 -= v w^T + w v^T, one warp per row
            for (int r = gwarp; r < L; r += nwarps) {
                double *row = A + (size_t)(k + 1 + r) * n + k + 1;
                const double vr = v[r], wr = w[r];
                for (int j = lane; j < L; j += 32) row[j] -= vr * w[j] + wr * v[j];
            }
        }
        grid.sync();
    }
    if (blockIdx.x == 0 && tid == 0) {
        d[n - 1] = A[(size_t)(n - 1) * n + (n - 1)];
        tau[n - 1] = 0.0;
    }
}

// A = (A + A^T) / 2 against the rounding of the products that gave it, and the
// largest biased exponent of its entries (out starts at zero).
__global__ void __launch_bounds__(kTriThreads) k_symmetrize_max(int n, double *__restrict__ A, int *__restrict__ out) {
    const int64_t idx = (int64_t)blockIdx.x * kTriThreads + threadIdx.x;
    const int i = (int)(idx / n), j = (int)(idx % n);
    int m = 0;
    if (i < n && j >= i) {
        double v = A[(size_t)i * n + j];
        if (j > i) {
            v = 0.5 * (v + A[(size_t)j * n + i]);
            A[(size_t)i * n + j] = v;
            A[(size_t)j * n + i] = v;
        }
        m = (__double2hiint(v) >> 20) & 0x7FF;
    }
    m = __reduce_max_sync(0xffffffffu, m);
    // most warps find it reached already
    if ((threadIdx.x & 31) == 0 && m > *(volatile int *)out) atomicMax(out, m);
}

// Power of two that brings a matrix with that exponent near 1; 0 where it is
// within 2^+-100 as it is (or holds infinities or NaN).
__device__ __forceinline__ int range_shift(int e) {
    const int q = 1023 - max(e, 1);
    return e == 0x7FF || abs(q) <= 100 ? 0 : q;
}
// Threads of k_tridiag_rows: one warp per SM sub-partition.  FP64 issues at a
// 64th of the FP32 rate here, so every FP64 instruction that all warps repeat
// (reductions, the reflector's scalars) costs its full issue time once per
// warp on a sub-partition; with one warp each that cost is paid once.
constexpr int kTrdThreads = 128;

// Sum over the warp in fixed point: every value as a 57-bit integer against the
// warp's largest exponent, three limbs added by redux, the total rounded once.
// An FP64 add of a warp costs 64 to 76 issue clocks and 106 through a shuffle, five of
// them 530; this takes about 200, and the values' truncation (2^-57 of the
// largest) stays below the rounding of the FP64 tree.
__device__ __forceinline__ double warp_sum_fixed(double v) {
    const int h = __double2hiint(v), e = (h >> 20) & 0x7FF;
    const int em = __reduce_max_sync(0xffffffffu, e);
    if (em == 0x7FF) {  // infinities and NaN
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        return v;
    }
    const unsigned long long M =
        ((unsigned long long)((unsigned)(h & 0xFFFFF) | (e ? 0x100000u : 0u)) << 32) | (unsigned)__double2loint(v);
    long long T = (long long)((M << 4) >> min(em - e, 63));
    if (h < 0) T = -T;
    const unsigned s0 = __reduce_add_sync(0xffffffffu, (unsigned)T & 0x3FFFFFu);
    const unsigned s1 = __reduce_add_sync(0xffffffffu, (unsigned)(T >> 22) & 0x3FFFFFu);
    const int s2 = (int)__reduce_add_sync(0xffffffffu, (unsigned)(int)(T >> 44));
    const double t = (double)(((long long)s2 << 44) + ((long long)s1 << 22) + (long long)s0);
    // 2^(max(em, 1) - 1075 - 4), in two exact steps near the ends of the range
    const int q = max(em, 1) - 1079, th = __double2hiint(t);
    const int te = ((th >> 20) & 0x7FF) + q;
    if (t == 0.0) return 0.0;
    return te > 0 && te < 0x7FF ? __hiloint2double(th + q * 0x100000, __double2loint(t)) : ldexp(t, q);
}

// named barriers of the two halves of a k_tridiag_rows block
template <int ID, int COUNT>
__device__ __forceinline__ void bar_sync() {
    asm volatile("bar.sync %0, %1;" ::"n"(ID), "n"(COUNT) : "memory");
}
template <int ID, int COUNT>
__device__ __forceinline__ void bar_arrive() {
    asm volatile("bar.arrive %0, %1;" ::"n"(ID), "n"(COUNT) : "memory");
}

// sum over the kTrdThreads threads of the computing half; result in all of them
__device__ __forceinline__ double block_sum128(double v, double *red) {
    v = warp_sum_fixed(v);
    bar_sync<1, kTrdThreads>();  // red may still be read from the previous call
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    bar_sync<1, kTrdThreads>();
    return (red[0] + red[1]) + (red[2] + red[3]);
}

// sums of N <= 16 values (a power of two) over the warp: half of them to the
// other lane at each of log2 N exchanges (N + 3 adds for 8, chain of five);
// returns that of value lane & (N - 1)
template <int N>
__device__ __forceinline__ double warp_sums(const double (&a)[N], int lane) {
    double h[N];
#pragma unroll
    for (int i = 0; i < N; ++i) h[i] = a[i];
#pragma unroll
    for (int w = N / 2; w > 0; w >>= 1) {
        const bool up = lane & w;
#pragma unroll
        for (int i = 0; i < w; ++i)
            h[i] = (up ? h[i + w] : h[i]) + __shfl_xor_sync(0xffffffffu, up ? h[i] : h[i + w], w);
    }
#pragma unroll
    for (int w = N; w < 32; w <<= 1) h[0] += __shfl_xor_sync(0xffffffffu, h[0], w);
    return h[0];
}

// Waiting for `target` arrivals at a counter that starts at zero.  It gives up
// after two seconds (false, *err set); the CTAs that then leave let the others
// run into the same limit.
__device__ __forceinline__ bool grid_wait(unsigned *counter, unsigned target, double *err) {
    unsigned long long t0 = 0;
    for (unsigned it = 0;; ++it) {
        unsigned c;
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(c) : "l"(counter) : "memory");
        if (c >= target) return true;
        if ((it & 1023u) == 1023u) {
            unsigned long long t;
            asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
            if (t0 == 0) t0 = t;
            else if (t - t0 > 2000000000ull) {
                *err = 1.0;
                return false;
            }
        }
    }
}

// NA rows of a k_tridiag_rows CTA (a: the first, from column k + 1 on, n apart):
// x += cb up + ca P, the sums of x y over the block's threads into redr[warp], the
// first row also to rb if that is not null.  The loads of a step stand before its
// stores, which the compiler could not tell apart from them.
template <int NA, int STRIDE>
__device__ __forceinline__ void rows_pass(int L, int n, double *a, const double *y, const double *up, const double *P,
                                          double t, double tpu, int r0, int G, double *rb, double (*redr)[STRIDE]) {
    const int tid = threadIdx.x, lane = tid & 31;
    constexpr int N2 = NA <= 1 ? 1 : NA <= 2 ? 2 : NA <= 4 ? 4 : NA <= 8 ? 8 : 16;
    double acc[N2], ca[NA], cb[NA];
#pragma unroll
    for (int i = 0; i < N2; ++i) acc[i] = 0.0;
#pragma unroll
    for (int i = 0; i < NA; ++i) {
        const double ur = up[r0 + i * G + 1];
        ca[i] = -(t * ur);
        cb[i] = fma(tpu, ur, -(t * P[r0 + i * G]));
    }
    int j = tid;
    for (; j + kTrdThreads < L; j += 2 * kTrdThreads) {
        const int j1 = j + kTrdThreads;
        const double y0 = y[j], y1 = y[j1], u0 = up[j + 2], u1 = up[j1 + 2], p0 = P[j + 1], p1 = P[j1 + 1];
        double x0[NA], x1[NA];
#pragma unroll
        for (int i = 0; i < NA; ++i) x0[i] = a[(size_t)i * n + j], x1[i] = a[(size_t)i * n + j1];
#pragma unroll
        for (int i = 0; i < NA; ++i) {
            x0[i] = fma(cb[i], u0, fma(ca[i], p0, x0[i]));
            x1[i] = fma(cb[i], u1, fma(ca[i], p1, x1[i]));
        }
#pragma unroll
        for (int i = 0; i < NA; ++i) {
            a[(size_t)i * n + j] = x0[i];
            a[(size_t)i * n + j1] = x1[i];
            acc[i] = fma(x1[i], y1, fma(x0[i], y0, acc[i]));
        }
        if (rb) rb[j] = x0[0], rb[j1] = x1[0];
    }
    if (j < L) {
        const double y0 = y[j], u0 = up[j + 2], p0 = P[j + 1];
        double x0[NA];
#pragma unroll
        for (int i = 0; i < NA; ++i) x0[i] = a[(size_t)i * n + j];
#pragma unroll
        for (int i = 0; i < NA; ++i) x0[i] = fma(cb[i], u0, fma(ca[i], p0, x0[i]));
#pragma unroll
        for (int i = 0; i < NA; ++i) {
            a[(size_t)i * n + j] = x0[i];
            acc[i] = fma(x0[i], y0, acc[i]);
        }
        if (rb) rb[j] = x0[0];
    }
    const double rs = warp_sums<N2>(acc, lane);
    if (lane < NA) redr[tid >> 5][lane] = rs;
}

// Tridiagonalisation with the matrix resident in shared memory.  CTA b owns
// the rows b, b + G, b + 2G, ... (full length n), so the product p = t A22 u
// and the rank-2 update of every column read and write only shared memory,
// and one grid barrier per column suffices: before it every CTA writes its
// entries of A22 y, y the column to reduce, and the owner of row k+1 writes that
// row as it stands before the update of column k; after it every CTA forms, from
// that row, the updated row k+1, which by symmetry is the next column to reduce.
// The update of column k is applied to the owned rows in the same pass as the
// product of column k+1.
//
// The reflector is I - t u u^T with u = y but for its first entry (u_0 = y_0 -
// beta, t = -1 / (beta u_0)): nothing is scaled, and A22 u = A22 y + (u_0 - y_0)
// A22 e_0, whose last vector is the row k+1 that every CTA receives.  So the
// product does not wait for the reflector: its norm, square root and reciprocal
// are computed while the entries travel.  t is about 1 / ||u||^2 and t (p.u) up to
// ||A|| / ||u||^2: A is brought near 1 by a power of two where it is not within
// 2^+-100 (as the rows are loaded; k_tri_prep takes it off T), and a column whose
// norm is below 2^-400 is taken as reduced (its entries below the first are
// dropped, a backward error of 2^-300 ||A|| at the most), so neither overflows.
// With p = t A22 u and w = p - (t/2)(p.u) u the update of row r is -(u_r w + w_r u) = -(u_r p + b_r u), b_r = p_r - t (p.u)
// u_r: w is not formed.  An entry costs three FP64 instructions.
// The second half of a block's threads only communicates: it arrives at the
// barrier, waits and brings the entries to shared memory.
// What bounds it: a chain per column.  Clocks at n = 75 / 750 (152 SMs): the rows
// 1,800 / 3,800 (FP64 issue, 2,900 of them at 750), the other warps' sums 260 / 500,
// then the reflector 2,600 / 3,200 (and some 300 for the square root and the division)
// beside the barrier and the loads 3,300 / 4,900, u^T A u 900 / 1,450, the next column
// 460 / 980.  Per column 3.5 us at 75 and 5.8 us at 750; with the reflector before the
// product, one thread polling and loading after it, and branches between the rows
// 4.6 and 7.4; with scaled reflectors, w formed, FP64 shuffles for the sums and
// divisions 8.1 at 750.  Entries tagged with their column and polled for by every
// thread, instead of the barrier, took 8,000 clocks per column at n = 750 (the
// polling loads themselves).
// Shared memory: R n (owned rows, R = ceil(n / G) <= RMAX) + 4 n doubles.
template <int RMAX>
__global__ void __launch_bounds__(2 * kTrdThreads) k_tridiag_rows(int n, const double *__restrict__ A, double *__restrict__ d,
                                                            double *__restrict__ e, double *__restrict__ tau,
                                                            double *__restrict__ Vh, double *__restrict__ pbuf,
                                                            double *__restrict__ rbuf, unsigned *__restrict__ counter,
                                                            double *__restrict__ err, const int *__restrict__ amax) {
    constexpr int NW = kTrdThreads / 32;
    extern __shared__ double sm[];
    const int G = gridDim.x, b = blockIdx.x, tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int R = (n - b + G - 1) / G;          // rows owned by this CTA
    const int Rmax = (n + G - 1) / G;
    double *rows = sm;                           // Rmax x n
    double *cur = rows + (size_t)Rmax * n;       // row k: cur[i] = A[k, k + i]; then u of column k in cur[1 + i]
    double *prev = cur + n;                      // the same of column k - 1
    double *P = prev + n, *tu = P + n;           // A u of column k - 1 (index 0 <-> row k); t u of column k
    __shared__ double red[NW];
    __shared__ double redr[NW][RMAX];
    __shared__ int gave_up;
    const int shift = range_shift(*amax);
    for (int i = 0; i < R; ++i) {
        const double *src = A + (size_t)(b + i * G) * n;
        for (int j = tid; j < n; j += 2 * kTrdThreads) rows[(size_t)i * n + j] = shift ? ldexp(src[j], shift) : src[j];
    }
    // no update before the first column: zeros in u and P of the one before
    for (int j = tid; j < n; j += 2 * kTrdThreads) cur[j] = shift ? ldexp(A[j], shift) : A[j], prev[j] = P[j] = 0.0;
    if (tid == 0) gave_up = 0;
    __syncthreads();
    if (tid >= kTrdThreads) {
        // communicating half
        const int lt = tid - kTrdThreads;
        for (int k = 0; k + 1 < n; ++k) {
            const int L = n - k - 1;
            const double *ab = pbuf + (size_t)(k & 1) * n, *rb = rbuf + (size_t)(k & 1) * n;
            bar_sync<2, 2 * kTrdThreads>();  // this CTA's entries are written, prev and P are free
            if (lt == 0) {
                asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(counter) : "memory");
                if (!grid_wait(counter, (unsigned)(k + 1) * (unsigned)G, err)) gave_up = 1;
            }
            bar_sync<3, kTrdThreads>();
            if (!gave_up) {
#pragma unroll 4
                for (int j = lt; j < L; j += kTrdThreads) {
                    const double rj = __ldcg(rb + j), aj = __ldcg(ab + j);
                    prev[j] = rj;
                    P[j] = aj;
                }
            }
            bar_sync<4, 2 * kTrdThreads>();
            if (gave_up) return;
            double *tmp = prev;
            prev = cur;
            cur = tmp;
        }
        return;
    }
    double tpu = 0.0, tp = 0.0;  // t (p.u), t of column k - 1
    for (int k = 0; k + 1 < n; ++k) {
        const int L = n - k - 1;
        const double x0 = cur[1];
        // owned rows r >= k + 1: update of column k - 1 on columns >= k + 1, then
        // the product with y = cur[1 .. L], the column below the diagonal
        const int i0 = k + 1 > b ? (k + 1 - b + G - 1) / G : 0, na = R - i0;
        double *ab = pbuf + (size_t)(k & 1) * n;
        {
            // row k + 1 is the first of its owner's rows that are left
            double *rb = b + i0 * G == k + 1 ? rbuf + (size_t)(k & 1) * n : nullptr;
            double *a = rows + (size_t)i0 * n + k + 1;
            const int r0 = b + i0 * G - k;
#define HSIM_ROWS(NA)                                                                              \
    case NA:                                                                                       \
        if (NA <= RMAX) rows_pass<NA <= RMAX ? NA : 1>(L, n, a, cur + 1, prev, P, tp, tpu, r0, G, rb, redr); \
        break
            switch (na) {
                HSIM_ROWS(1);
                HSIM_ROWS(2);
                HSIM_ROWS(3);
                HSIM_ROWS(4);
                HSIM_ROWS(5);
                HSIM_ROWS(6);
                HSIM_ROWS(7);
                HSIM_ROWS(8);
                HSIM_ROWS(9);
                HSIM_ROWS(10);
                HSIM_ROWS(11);
                HSIM_ROWS(12);
                HSIM_ROWS(13);
                HSIM_ROWS(14);
                HSIM_ROWS(15);
                HSIM_ROWS(16);
                default: break;  // none left
            }
#undef HSIM_ROWS
        }
        bar_sync<1, kTrdThreads>();
        if (tid < na)
            ab[b + (i0 + tid) * G - k - 1] = (redr[0][tid] + redr[1][tid]) + (redr[2][tid] + redr[3][tid]);
        bar_arrive<2, 2 * kTrdThreads>();
        // meanwhile the reflector
        double part = 0.0;
        for (int i = 1 + tid; i < L; i += kTrdThreads) part = fma(cur[1 + i], cur[1 + i], part);
        const double sigma = block_sum128(part, red);
        double beta = x0, t = 0.0, u0 = 1.0;
        // (tests on the bits: an FP64 comparison waits for the pipe)
        if ((__double2hiint(sigma) | __double2loint(sigma)) != 0) {
            const double s2 = fma(x0, x0, sigma);
            if (((__double2hiint(s2) >> 20) & 0x7FF) >= 1023 - 800) {
                const double mu = sqrt(s2);
                beta = __double2hiint(x0) >= 0 ? -mu : mu;
                u0 = x0 - beta;
                t = -1.0 / (beta * u0);
            }
        }
        const double d0 = u0 - x0, c0 = u0 * t;
        for (int i = tid; i < L; i += kTrdThreads) {
            const double ui = i == 0 ? u0 : cur[1 + i];
            if (i == 0) cur[1] = u0;
            tu[i] = t * ui;
            if (b == 0) Vh[(size_t)k * n + k + 1 + i] = ui;
        }
        if (b == 0 && tid == 0) {
            d[k] = cur[0];
            e[k] = beta;
            tau[k] = t;
        }
        bar_sync<4, 2 * kTrdThreads>();
        if (gave_up) return;
        // P = A u from A y (in P), and row k + 1 (in prev) after the update of
        // column k
        double pu = 0.0;
        int j = tid;
        for (; j + kTrdThreads < L; j += 2 * kTrdThreads) {
            const int j1 = j + kTrdThreads;
            const double a0 = P[j], a1 = P[j1], r0 = prev[j], r1 = prev[j1], t0 = tu[j], t1 = tu[j1];
            const double P0 = fma(d0, r0, a0), P1 = fma(d0, r1, a1);
            P[j] = P0, P[j1] = P1;
            pu = fma(P1, t1, fma(P0, t0, pu));
        }
        if (j < L) {
            const double P0 = fma(d0, prev[j], P[j]);
            P[j] = P0;
            pu = fma(P0, tu[j], pu);
        }
        tpu = t * block_sum128(pu, red);
        const double b0 = fma(-tpu, u0, t * P[0]);
        for (j = tid; j + kTrdThreads < L; j += 2 * kTrdThreads) {
            const int j1 = j + kTrdThreads;
            const double a0 = P[j], a1 = P[j1], r0 = prev[j], r1 = prev[j1], v0 = cur[1 + j], v1 = cur[1 + j1];
            prev[j] = fma(-b0, v0, fma(-c0, a0, r0));
            prev[j1] = fma(-b0, v1, fma(-c0, a1, r1));
        }
        if (j < L) prev[j] = fma(-b0, cur[1 + j], fma(-c0, P[j], prev[j]));
        tp = t;
        double *tmp = prev;
        prev = cur;
        cur = tmp;
        bar_sync<1, kTrdThreads>();
    }
    if (b == 0 && tid == 0) {
        d[n - 1] = cur[0];
        tau[n - 1] = 0.0;
    }
}

// Compact WY of every block of eight consecutive reflectors k0 .. k0 + 7: H_k0 ...
// H_{k0+7} = I - V T V^T, T (8 x 8, upper triangular, row-major) from the Gram
// matrix of the block's vectors.  One CTA per block.
constexpr int kWY = 8;
__global__ void __launch_bounds__(128) k_tri_wy(int n, const double *__restrict__ Vh, const double *__restrict__ tau,
                                                double *__restrict__ Tw) {
    __shared__ double G[kWY][kWY], T[kWY][kWY];
    const int k0 = blockIdx.x * kWY, lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    // pairs (i, j), i < j: dot over the rows where both are stored (j's)
    for (int q = wid; q < kWY * kWY; q += 4) {
        const int i = q / kWY, j = q % kWY;
        if (i >= j) continue;
        double s = 0.0;
        if (k0 + j < n - 1) {
            const double *vi = Vh + (size_t)(k0 + i) * n, *vj = Vh + (size_t)(k0 + j) * n;
            for (int r = k0 + j + 1 + lane; r < n; r += 32) s = fma(vi[r], vj[r], s);
            s = warp_sum_fixed(s);
        }
        if (lane == 0) G[i][j] = s;
    }
    __syncthreads();
    if (threadIdx.x < kWY) {
        const int r = threadIdx.x;  // row of T
        for (int i = 0; i < kWY; ++i) {
            const double t = k0 + i < n - 1 ? tau[k0 + i] : 0.0;
            double v = r == i ? t : 0.0;
            if (r < i) {
                double s = 0.0;
                for (int j = r; j < i; ++j) s = fma(T[r][j], G[j][i], s);
                v = -t * s;
            }
            T[r][i] = v;
            __syncwarp(0xffu);
        }
    }
    __syncthreads();
    if (threadIdx.x < kWY * kWY) Tw[(size_t)blockIdx.x * kWY * kWY + threadIdx.x] = T[threadIdx.x / kWY][threadIdx.x % kWY];
}

// Back transformation X = Q Z with Q = H_0 H_1 ... H_{n-2}, eight reflectors at a
// time (last block first): z -= V (T (V^T z)).  A CTA holds nv <= NV vectors in
// registers, thread t the rows t, t + 128, ...; the block's V is staged in shared
// memory while the block before is applied.
// What bounds it: FP64 instructions, 2 x nv x rows / 128 per reflector and warp,
// balanced over the SMs (nv = m / SMs).  n = m = 750: 1.35 ms (2.9
// with a fixed-point sum per dot product); one warp per vector and one reflector
// at a time took 2.2 ms (750 warps on 608 sub-partitions, five FP64 adds for the
// sum and a barrier per reflector).
template <int RPT, int NV>
__global__ void __launch_bounds__(128) k_tri_back_wy(int n, int m, int nv, int bufs, const double *__restrict__ Vh,
                                                     const double *__restrict__ Tw, const double *__restrict__ Z,
                                                     double *__restrict__ X, int ldx) {
    extern __shared__ double vs[];  // bufs (1 or 2) buffers of kWY x n
    __shared__ double red[4][kWY * NV], cs[kWY * NV], Ts[2][kWY * kWY];
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int i0 = blockIdx.x * nv, cnt = min(nv, m - i0);
    double z[NV][RPT];
#pragma unroll
    for (int v = 0; v < NV; ++v)
#pragma unroll
        for (int q = 0; q < RPT; ++q) {
            const int j = tid + 128 * q;
            z[v][q] = v < cnt && j < n ? Z[(size_t)(i0 + v) * n + j] : 0.0;
        }
    const int nb = (n - 1 + kWY - 1) / kWY;
    // rows j > k of reflector k, zero elsewhere
    auto stage = [&](int b, int buf) {
        double *dst = vs + (size_t)buf * kWY * n;
        // from the first row of 128 that the block touches
        for (int kk = 0; kk < kWY; ++kk) {
            const int k = b * kWY + kk;
            for (int j = ((b * kWY + 1) & ~127) + tid; j < n; j += 128) {
                const bool live = k < n - 1 && j > k;
                const unsigned d = (unsigned)__cvta_generic_to_shared(dst + kk * n + j);
                asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;\n" ::"r"(d),
                             "l"(Vh + (live ? (size_t)k * n + j : 0)), "r"(live ? 8 : 0));
            }
        }
        if (tid < kWY * kWY) Ts[buf][tid] = Tw[(size_t)b * kWY * kWY + tid];
        asm volatile("cp.async.commit_group;\n" ::: "memory");
    };
    if (bufs == 2) stage(nb - 1, (nb - 1) & 1);
    for (int b = nb - 1; b >= 0; --b) {
        const int cur = bufs == 2 ? b & 1 : 0;
        if (bufs == 1) stage(b, 0);
        else if (b > 0) stage(b - 1, cur ^ 1);
        if (bufs == 2 && b > 0) asm volatile("cp.async.wait_group 1;\n" ::: "memory");
        else asm volatile("cp.async.wait_group 0;\n" ::: "memory");
        __syncthreads();
        const double *V = vs + (size_t)cur * kWY * n;
        const int q0 = (b * kWY + 1) >> 7;  // rows below are zero in the whole block
        double s[kWY][NV];
#pragma unroll
        for (int kk = 0; kk < kWY; ++kk)
#pragma unroll
            for (int v = 0; v < NV; ++v) s[kk][v] = 0.0;
#pragma unroll
        for (int q = 0; q < RPT; ++q) {
            const int j = tid + 128 * q;
            if (q < q0 || 128 * q >= n) continue;
#pragma unroll
            for (int kk = 0; kk < kWY; ++kk) {
                const double x = j < n ? V[kk * n + j] : 0.0;
#pragma unroll
                for (int v = 0; v < NV; ++v) s[kk][v] = fma(x, z[v][q], s[kk][v]);
            }
        }
        // half of the reflectors to the other lane at each of three exchanges
        // (7 adds per vector in place of 24), reflector lane & 7 is left
#pragma unroll
        for (int v = 0; v < NV; ++v) {
            double h4[4], h2[2], h1;
            const bool b4 = lane & 4, b2 = lane & 2, b1 = lane & 1;
#pragma unroll
            for (int u = 0; u < 4; ++u)
                h4[u] = (b4 ? s[u + 4][v] : s[u][v]) + __shfl_xor_sync(0xffffffffu, b4 ? s[u][v] : s[u + 4][v], 4);
#pragma unroll
            for (int u = 0; u < 2; ++u)
                h2[u] = (b2 ? h4[u + 2] : h4[u]) + __shfl_xor_sync(0xffffffffu, b2 ? h4[u] : h4[u + 2], 2);
            h1 = (b1 ? h2[1] : h2[0]) + __shfl_xor_sync(0xffffffffu, b1 ? h2[0] : h2[1], 1);
            h1 += __shfl_xor_sync(0xffffffffu, h1, 8);
            h1 += __shfl_xor_sync(0xffffffffu, h1, 16);
            if (lane < kWY) red[wid][lane * NV + v] = h1;
        }
        __syncthreads();
        if (tid < kWY * NV) red[0][tid] = (red[0][tid] + red[1][tid]) + (red[2][tid] + red[3][tid]);
        __syncthreads();
        if (tid < kWY * NV) {
            const int i = tid / NV, v = tid % NV;
            double c = 0.0;
            for (int j = i; j < kWY; ++j) c = fma(Ts[cur][i * kWY + j], red[0][j * NV + v], c);
            cs[tid] = -c;
        }
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < kWY; ++kk) {
            double c[NV];
#pragma unroll
            for (int v = 0; v < NV; ++v) c[v] = cs[kk * NV + v];
#pragma unroll
            for (int q = 0; q < RPT; ++q) {
                const int j = tid + 128 * q;
                if (q < q0 || 128 * q >= n) continue;
                const double x = j < n ? V[kk * n + j] : 0.0;
#pragma unroll
                for (int v = 0; v < NV; ++v) z[v][q] = fma(c[v], x, z[v][q]);
            }
        }
        __syncthreads();  // before this buffer is staged again
    }
#pragma unroll
    for (int v = 0; v < NV; ++v)
#pragma unroll
        for (int q = 0; q < RPT; ++q) {
            const int j = tid + 128 * q;
            if (v < cnt && j < n) X[(size_t)j * ldx + i0 + v] = z[v][q];
        }
}

// T scaled by a power of two to a norm bound in [1/2, 1): ds, e2s = e^2 (at least
// 2^-120 in FP64 and 2^-40 in FP32: couplings of 2^-60 and 2^-20 of ||T||, below
// the accuracy of either count) and their FP32 copies; bounds: the Gershgorin
// interval of the scaled T, ||T|| (not scaled), the scale; F_j for k_tri_vectors
// amax (may be null): d and e come from a matrix scaled by 2^range_shift, which
// is taken off first.
__global__ void k_tri_prep(int n, double *__restrict__ d, double *__restrict__ e, const int *__restrict__ amax,
                           double *__restrict__ ds, double *__restrict__ e2s, double *__restrict__ bounds,
                           float *__restrict__ d32, float *__restrict__ e232, double *__restrict__ fm,
                           double *__restrict__ fi, int *__restrict__ fx) {
    __shared__ double red[3][kTriThreads / 32];
    __shared__ double sm[2][kTriThreads];
    __shared__ int sx[2][kTriThreads];
    const int shift = amax ? range_shift(*amax) : 0;
    if (shift) {
        for (int j = threadIdx.x; j < n; j += kTriThreads) {
            d[j] = ldexp(d[j], -shift);
            if (j + 1 < n) e[j] = ldexp(e[j], -shift);
        }
        __syncthreads();
    }
    double lo = DBL_MAX, hi = -DBL_MAX, nm = 0.0;
    for (int j = threadIdx.x; j < n; j += kTriThreads) {
        const double r = (j > 0 ? fabs(e[j - 1]) : 0.0) + (j + 1 < n ? fabs(e[j]) : 0.0);
        lo = fmin(lo, d[j] - r);
        hi = fmax(hi, d[j] + r);
        nm = fmax(nm, fabs(d[j]) + r);
    }
    for (int o = 16; o > 0; o >>= 1) {
        lo = fmin(lo, __shfl_xor_sync(0xffffffffu, lo, o));
        hi = fmax(hi, __shfl_xor_sync(0xffffffffu, hi, o));
        nm = fmax(nm, __shfl_xor_sync(0xffffffffu, nm, o));
    }
    const int w = threadIdx.x >> 5;
    if ((threadIdx.x & 31) == 0) {
        red[0][w] = lo;
        red[1][w] = hi;
        red[2][w] = nm;
    }
    __syncthreads();
    for (int i = 0; i < kTriThreads / 32; ++i) {
        lo = fmin(lo, red[0][i]);
        hi = fmax(hi, red[1][i]);
        nm = fmax(nm, red[2][i]);
    }
    int ex = 0;
    if (nm > 0.0 && nm <= DBL_MAX) frexp(nm, &ex);
    const double sc = ldexp(1.0, min(max(-ex, -1000), 1000));
    for (int j = threadIdx.x; j < n; j += kTriThreads) {
        ds[j] = d[j] * sc;
        d32[j] = (float)(d[j] * sc);
        if (j + 1 < n) {
            const double es = e[j] * sc, q = es * es;
            e2s[j] = fmax(q, 0x1p-120);
            e232[j] = fmaxf((float)q, 0x1p-40f);
        }
    }
    // F_j = prod_{i < j} (-e_i) of the scaled T as fm 2^fx (fi = 1 / fm): every
    // thread a run of factors, then a scan over the runs
    const int run = (n + kTriThreads - 1) / kTriThreads, j0 = min(n, (int)threadIdx.x * run), j1 = min(n, j0 + run);
    auto norm = [](double &m, int &x) {
        const int h = __double2hiint(m), q = ((h >> 20) & 0x7FF) - 1023;
        m = __hiloint2double(h - q * 0x100000, __double2loint(m));
        x += q;
    };
    auto factor = [&](int i) {
        const double es = i + 1 < n ? e[i] * sc : 1.0;
        return -copysign(fmax(fabs(es), 0x1p-60), es);
    };
    double pm = 1.0;
    int px = 0;
    for (int i = j0; i < j1; ++i) {
        pm *= factor(i);
        norm(pm, px);
    }
    int cur = 0;
    sm[0][threadIdx.x] = pm;
    sx[0][threadIdx.x] = px;
    __syncthreads();
    for (int o = 1; o < kTriThreads; o <<= 1) {
        if ((int)threadIdx.x >= o) {
            pm *= sm[cur][threadIdx.x - o];
            px += sx[cur][threadIdx.x - o];
            norm(pm, px);
        }
        cur ^= 1;
        sm[cur][threadIdx.x] = pm;
        sx[cur][threadIdx.x] = px;
        __syncthreads();
    }
    pm = threadIdx.x > 0 ? sm[cur][threadIdx.x - 1] : 1.0;
    px = threadIdx.x > 0 ? sx[cur][threadIdx.x - 1] : 0;
    for (int i = j0; i < j1; ++i) {
        fm[i] = pm;
        fi[i] = 1.0 / pm;
        fx[i] = px;
        pm *= factor(i);
        norm(pm, px);
    }
    if (threadIdx.x == 0) {
        const double pad = 4.0 * DBL_EPSILON;
        bounds[0] = lo * sc - pad;
        bounds[1] = hi * sc + pad;
        bounds[2] = nm;
        bounds[3] = sc;
    }
}

// Eigenvalues of the scaled T below x, and det(T - x I) as fm 2^fe.  The Sturm
// sequence p_{j+1} = (d_j - x) p_j - e_j^2 p_{j-1} without divisions: three FP64
// instructions a step, where d - x - e^2 / q takes about ten, and an FP64
// instruction of a warp issues every 64 to 76 clocks on a sub-partition.  The count is
// the number of sign changes (an exact zero is counted with its own or the next
// step, whatever its sign).  |d - x| <= 2, 2^-120 <= e^2 <= 1: eight steps grow
// p by at most 2^13 and shrink it by at most 2^-480, then the pair is rescaled
// by its exponent.
__device__ __forceinline__ int sturm_count(int n, const double *__restrict__ d, const double *__restrict__ e2,
                                           double x, double &fm, int &fe) {
    double p0 = 1.0, p1 = d[0] - x;
    unsigned h1 = (unsigned)__double2hiint(p1);
    int c = h1 >> 31, E = 0;
    auto step = [&](double dj, double ej) {
        const double p2 = fma(dj - x, p1, -(ej * p0));
        const unsigned h2 = (unsigned)__double2hiint(p2);
        c += (h2 ^ h1) >> 31;
        p0 = p1;
        p1 = p2;
        h1 = h2;
    };
    for (int j = 1; j < n;) {
        if (j + 8 <= n) {
            double dj[8], ej[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) dj[u] = d[j + u], ej[u] = e2[j + u - 1];
#pragma unroll
            for (int u = 0; u < 8; ++u) step(dj[u], ej[u]);
            j += 8;
        } else {
            for (; j < n; ++j) step(d[j], e2[j - 1]);
        }
        const int e0 = (__double2hiint(p0) >> 20) & 0x7FF, e1 = (__double2hiint(p1) >> 20) & 0x7FF;
        const int sh = max(e0, e1) - 1023;
        // entries 2^-1000 below the larger one become zero (with their sign)
        p0 = __hiloint2double(e0 > sh ? __double2hiint(p0) - sh * 0x100000 : __double2hiint(p0) & 0x80000000,
                              e0 > sh ? __double2loint(p0) : 0);
        p1 = __hiloint2double(e1 > sh ? __double2hiint(p1) - sh * 0x100000 : __double2hiint(p1) & 0x80000000,
                              e1 > sh ? __double2loint(p1) : 0);
        E += sh;
    }
    fm = p1;
    fe = E;
    return c;
}

// the same in FP32 (e^2 >= 2^-40, rescaled every four steps), for brackets of
// 1e-5 ||T||
__device__ __forceinline__ int sturm_count32(int n, const float *__restrict__ d, const float *__restrict__ e2, float x) {
    float p0 = 1.f, p1 = d[0] - x;
    unsigned h1 = __float_as_uint(p1);
    int c = h1 >> 31;
    auto step = [&](float dj, float ej) {
        const float p2 = fmaf(dj - x, p1, -(ej * p0));
        const unsigned h2 = __float_as_uint(p2);
        c += (h2 ^ h1) >> 31;
        p0 = p1;
        p1 = p2;
        h1 = h2;
    };
    for (int j = 1; j < n;) {
        if (j + 4 <= n) {
            float dj[4], ej[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) dj[u] = d[j + u], ej[u] = e2[j + u - 1];
#pragma unroll
            for (int u = 0; u < 4; ++u) step(dj[u], ej[u]);
            j += 4;
        } else {
            for (; j < n; ++j) step(d[j], e2[j - 1]);
        }
        const int e0 = (__float_as_uint(p0) >> 23) & 0xFF, e1 = (h1 >> 23) & 0xFF;
        const int sh = max(e0, e1) - 127;
        p0 = __uint_as_float(e0 > sh ? __float_as_uint(p0) - (unsigned)(sh * 0x800000) : __float_as_uint(p0) & 0x80000000u);
        p1 = __uint_as_float(e1 > sh ? h1 - (unsigned)(sh * 0x800000) : h1 & 0x80000000u);
        h1 = __float_as_uint(p1);
    }
    return c;
}

// number of leading lanes of the group whose count is at most i (monotone up to
// rounding: the highest such lane decides)
__device__ __forceinline__ int group_le(bool le, int gbase, int L) {
    const unsigned bal = __ballot_sync(0xffffffffu, le);
    const unsigned g = (L == 32) ? bal : (bal >> gbase) & ((1u << L) - 1u);
    return g == 0 ? 0 : 32 - __clz(g);
}

// lambda_i, i < m: G eigenvalues per warp, L = 32 / G >= 2 lanes each, every
// lane a Sturm count per round.  FP32 multisection down to 1e-5 ||T||; a first
// FP64 round on points from end to end of that bracket, which is widened until
// its counts hold; then FP64 rounds to full precision.  Where the bracket holds
// the one eigenvalue, the lanes gather around the zero of the chord of the
// determinant, at distances of 2^-3 to 2^-24 of the bracket on either side: the
// chord is off by about (bracket / gap) brackets, so the bracket shrinks
// quadratically (three to four FP64 rounds at n = 750, where equal sections take
// nine); the counts still decide, and a round that does not shrink the bracket
// fourfold, or a bracket of several eigenvalues, is followed by equal sections.
// What bounds it: an FP64 round is n dependent steps of three instructions of 64 to 76
// clocks, 84 us at n = 750 with one warp per sub-partition (G = ceil(m / (4 SMs)):
// a second warp on a sub-partition doubles every round).
__global__ void k_tri_bisect(int n, int m, int G, const double *__restrict__ d, const double *__restrict__ e2,
                             const float *__restrict__ d32, const float *__restrict__ e232,
                             const double *__restrict__ bounds, double *__restrict__ lam) {
    const int lane = threadIdx.x & 31, warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int L = 32 / G, gi = lane / L, li = lane % L, gbase = gi * L;
    const int i = warp * G + gi;
    const bool valid = gi < G && i < m;
    if (warp * G >= m) return;  // uniform per warp
    const double glo = bounds[0], ghi = bounds[1], tn = bounds[2] * bounds[3];
    const double sect = 1.0 / (L + 1);
    double lo = glo, hi = ghi;
    for (int round = 0; round < 64; ++round) {
        const bool go = valid && hi - lo > 1e-5;
        if (!__any_sync(0xffffffffu, go)) break;
        const double x = lo + (hi - lo) * ((li + 1) * sect);
        const bool le = go && sturm_count32(n, d32, e232, (float)x) <= i;
        const int nle = group_le(le, gbase, L);
        if (go) {
            const double nlo = nle > 0 ? lo + (hi - lo) * (nle * sect) : lo;
            const double nhi = nle < L ? lo + (hi - lo) * ((nle + 1) * sect) : hi;
            lo = nlo;
            hi = nhi;
        }
    }
    // one FP64 round of the whole warp: counts at x (ascending lanes of a group)
    // move lo and hi; flo, fhi: the determinant there (fe < kNone: not known),
    // clo, chi: the counts
    constexpr int kNone = -(1 << 30);
    double flo = 0.0, fhi = 0.0;
    int elo = kNone, ehi = kNone, clo = 0, chi = 0;
    auto narrow = [&](double x, bool go) {
        double fm = 0.0;
        int fe = 0;
        const int cnt = go ? sturm_count(n, d, e2, x, fm, fe) : 0;
        const int nle = group_le(go && cnt <= i, gbase, L);
        const int sl = gbase + max(nle - 1, 0), sh = gbase + min(nle, L - 1);
        const double xl = __shfl_sync(0xffffffffu, x, sl & 31), xh = __shfl_sync(0xffffffffu, x, sh & 31);
        const double ml = __shfl_sync(0xffffffffu, fm, sl & 31), mh = __shfl_sync(0xffffffffu, fm, sh & 31);
        const int fl = __shfl_sync(0xffffffffu, fe, sl & 31), fh = __shfl_sync(0xffffffffu, fe, sh & 31);
        const int cl = __shfl_sync(0xffffffffu, cnt, sl & 31), ch = __shfl_sync(0xffffffffu, cnt, sh & 31);
        if (go && nle > 0) lo = xl, flo = ml, elo = fl, clo = cl;
        if (go && nle < L) hi = xh, fhi = mh, ehi = fh, chi = ch;
        return nle;
    };
    // the FP32 bracket, end to end; widened where its own ends do not hold
    double wid = fmax(hi - lo, 1e-5);
    bool checked = !valid;
    for (int t = 0; t < 64; ++t) {
        if (!__any_sync(0xffffffffu, !checked)) break;
        const double l0 = lo, h0 = hi;
        const int nle = narrow(l0 + (h0 - l0) * ((double)li / (L - 1)), !checked);
        if (!checked) {
            const bool okl = nle > 0 || l0 <= glo, okh = nle < L || h0 >= ghi;
            checked = okl && okh;
            if (!okl) lo = fmax(glo, l0 - wid), hi = l0, elo = kNone;
            if (!okh) hi = fmin(ghi, h0 + wid), lo = h0, ehi = kNone;
            wid *= 2.0;
        }
    }
    // to 2 eps (|lambda| + ||T||), the absolute accuracy of a dense symmetric
    // eigensolve (a quarter of it: a round more, the vectors' error unchanged)
    const int H = L / 2;
    bool chord = true;
    for (int round = 0; round < 200; ++round) {
        const double w = hi - lo, mid = lo + 0.5 * w;
        const bool go = valid && !(w <= 2.0 * DBL_EPSILON * (tn + fmax(fabs(lo), fabs(hi))) || mid <= lo || mid >= hi);
        if (!__any_sync(0xffffffffu, go)) break;
        double x = lo + w * ((li + 1) * sect);
        const bool one = L >= 8 && chord && elo != kNone && ehi != kNone && clo == i && chi == i + 1;
        if (one) {
            // |f(hi) / f(lo)| in FP32: the chord's zero to 24 bits of the bracket
            const int de = ehi - elo;
            const float r = fabsf((float)fhi / (float)flo) * exp2f((float)min(max(de, -100), 100));
            const double z = lo + w * (double)(1.f / (1.f + r));
            const int k = li < H ? li + 1 : L - li;  // 1 .. H from the outside in
            const double dl = w * (double)exp2f(-(float)(24 * k / H));
            x = fmin(fmax(li < H ? z - dl : z + dl, lo), hi);
        }
        narrow(x, go);
        chord = !one || !(hi - lo > 0.25 * w);
    }
    if (valid && li == 0) lam[i] = (lo + 0.5 * (hi - lo)) / bounds[3];
}

// uniform in [-1, 1) from a 64-bit hash (splitmix64 finaliser)
__device__ __forceinline__ double hash_uniform(uint64_t x) {
    x += 0x9E3779B97F4A7C15ull;
    x = (x ^ (x >> 30)) * 0xBF58476D1CE4E5B9ull;
    x = (x ^ (x >> 27)) * 0x94D049BB133111EBull;
    x ^= x >> 31;
    return (double)(x >> 11) * (2.0 / 9007199254740992.0) - 1.0;
}

__device__ __forceinline__ double warp_sum(double v) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Eigenvectors of T for single eigenvalues: column k of the adjugate of T -
// lambda I,
//     z_j = P_j prod_{i=j}^{k-1} (-e_i) B_{k+1}  (j <= k),
//     z_j = P_k prod_{i=k}^{j-1} (-e_i) B_{j+1}  (j > k),
// P_j and B_j the determinants of the leading j rows and of the rows from j on,
// k where |P_k B_{k+1}| is largest (the diagonal of the adjugate goes with the
// squares of the vector's entries; the twisted factorisation of Dhillon and
// Parlett in product form).  One vector of inverse iteration with LU cost two
// dependent divisions a step and three solves, one lane at work (1.32 ms for 750
// vectors); here the two sequences run without divisions, sixteen vectors to a
// warp (forward in the lower lanes, backward in the upper: an FP64 instruction
// of a warp takes the same time for one lane as for 32), 0.1 ms.
//
// k_tri_minors: S_t = P_t (dir 0) and B_{n-t} (dir 1), t < n, as seq[dir][t][i]
// 2^xs[dir][t / 8][i]
__global__ void __launch_bounds__(32) k_tri_minors(int n, int m, const double *__restrict__ d, const double *__restrict__ e2,
                                                   const double *__restrict__ bounds, const double *__restrict__ lam,
                                                   double *__restrict__ seq, int *__restrict__ xs) {
    const int lane = threadIdx.x, i = blockIdx.x * 16 + (lane & 15), dir = lane >> 4;
    if (i >= m) return;
    const double x = lam[i] * bounds[3];
    double *out = seq + (size_t)dir * n * m + i;
    int *ox = xs + (size_t)dir * ((n + 7) / 8) * m + i;
    // step t: row t forward, n - 1 - t backward, coupled by e2[t - 1] or e2[n - 1 - t]
    const double *dp = dir ? d + (n - 1) : d;
    const double *ep = dir ? e2 + (n - 1) : e2 - 1;
    const int sg = dir ? -1 : 1;
    double p0 = 0.0, p1 = 1.0;  // S_{t-1}, S_t
    int E = 0;
    for (int t = 0; t < n; t += 8) {
        ox[(size_t)(t >> 3) * m] = E;
        const int cnt = min(8, n - t);
        double dj[8], ej[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            dj[u] = u < cnt ? dp[sg * (t + u)] : 0.0;
            ej[u] = u < cnt && t + u > 0 ? ep[sg * (t + u)] : 0.0;
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            if (u >= cnt) break;
            out[(size_t)(t + u) * m] = p1;
            const double p2 = fma(dj[u] - x, p1, -(ej[u] * p0));
            p0 = p1;
            p1 = p2;
        }
        const int e0 = (__double2hiint(p0) >> 20) & 0x7FF, e1 = (__double2hiint(p1) >> 20) & 0x7FF;
        const int sh = max(e0, e1) - 1023;
        p0 = e0 > sh ? __hiloint2double(__double2hiint(p0) - sh * 0x100000, __double2loint(p0)) : 0.0;
        p1 = e1 > sh ? __hiloint2double(__double2hiint(p1) - sh * 0x100000, __double2loint(p1)) : 0.0;
        E += sh;
    }
}

// x 2^e, 0 below the normal range (entries 2^-1000 of the largest)
__device__ __forceinline__ double shift_exp(double x, int e) {
    const int h = __double2hiint(x), q = ((h >> 20) & 0x7FF) + e;
    return q > 0 && (h & 0x7FF00000) != 0 ? __hiloint2double(h + min(e, 4000) * 0x100000, __double2loint(x)) : 0.0;
}

// z for 8 vectors per CTA, thread (vector tid % 8, rows tid / 8, + 32, ...)
__global__ void __launch_bounds__(256) k_tri_vectors(int n, int m, const double *__restrict__ seq,
                                                     const int *__restrict__ xs, const double *__restrict__ fm,
                                                     const double *__restrict__ fi, const int *__restrict__ fx,
                                                     double *__restrict__ Z) {
    __shared__ float key[32][8];
    __shared__ int row[32][8];
    __shared__ double part[32][8];
    const int v = threadIdx.x & 7, r = threadIdx.x >> 3, i = blockIdx.x * 8 + v, nb = (n + 7) / 8;
    const bool ok = i < m;
    const double *P = seq + i, *B = seq + (size_t)n * m + i;
    const int *xP = xs + i, *xB = xs + (size_t)nb * m + i;
    // S^b_{n-1-j} = B_{j+1}
    auto lg = [](double x) {
        const int h = __double2hiint(x) & 0x7FFFFFFF;
        return h < 0x00100000 ? -3e38f : (float)((h >> 20) - 1023) + __log2f(__int_as_float(0x3F800000 | ((h & 0xFFFFF) << 3)));
    };
    float best = -3.4e38f;
    int k = 0;
    if (ok)
        for (int j = r; j < n; j += 32) {
            const int tb = n - 1 - j;
            const float q = lg(P[(size_t)j * m]) + lg(B[(size_t)tb * m]) + (float)(xP[(size_t)(j >> 3) * m] + xB[(size_t)(tb >> 3) * m]);
            if (q > best) best = q, k = j;
        }
    key[r][v] = best;
    row[r][v] = k;
    __syncthreads();
    for (int q = 0; q < 32; ++q)
        if (key[q][v] > best || (key[q][v] == best && row[q][v] < k)) best = key[q][v], k = row[q][v];
    double c1 = 0.0, c2 = 0.0;
    int s1 = 0, s2 = 0;
    if (ok) {
        const int tb = n - 1 - k;
        c1 = fm[k] / P[(size_t)k * m];
        c2 = fi[k] / B[(size_t)tb * m];
        s1 = fx[k] - xP[(size_t)(k >> 3) * m];
        s2 = -fx[k] - xB[(size_t)(tb >> 3) * m];
    }
    auto entry = [&](int j) {
        if (j <= k) return shift_exp(P[(size_t)j * m] * fi[j] * c1, xP[(size_t)(j >> 3) * m] - fx[j] + s1);
        const int tb = n - 1 - j;
        return shift_exp(B[(size_t)tb * m] * fm[j] * c2, xB[(size_t)(tb >> 3) * m] + fx[j] + s2);
    };
    double sum = 0.0;
    if (ok)
        for (int j = r; j < n; j += 32) {
            const double z = entry(j);
            sum = fma(z, z, sum);
        }
    part[r][v] = sum;
    __syncthreads();
    sum = 0.0;
#pragma unroll
    for (int q = 0; q < 32; ++q) sum += part[q][v];
    const double inv = rsqrt(sum);
    if (ok)
        for (int j = r; j < n; j += 32) Z[(size_t)i * n + j] = entry(j) * inv;
}

// Clusters: inverse iteration, one warp per cluster [cl[2 c], cl[2 c + 1]); Z is m x n
// (vector-major); LU scratch: 5 n doubles + n flags per cluster
__global__ void k_tri_invit(int n, const double *__restrict__ d, const double *__restrict__ e,
                            const double *__restrict__ bounds, const double *__restrict__ lam,
                            const int *__restrict__ cl, double *__restrict__ Z, double *__restrict__ scratch,
                            unsigned char *__restrict__ pivflag) {
    const int c = blockIdx.x, lane = threadIdx.x;
    const int i0 = cl[2 * c], i1 = cl[2 * c + 1];
    double *u0i = scratch + (size_t)c * 5 * n;  // reciprocal of the pivot
    double *u1 = u0i + n, *u2 = u1 + n, *l = u2 + n, *y = l + n;
    unsigned char *piv = pivflag + (size_t)c * n;
    const double small = DBL_EPSILON * fmax(bounds[2], DBL_MIN);
    for (int i = i0; i < i1; ++i) {
        double *z = Z + (size_t)i * n;
        const double lmb = lam[i];
        if (lane == 0) {
            // T - lmb I = P L U, U with three diagonals (u0, u1, u2)
            double cd = d[0] - lmb, cu = n > 1 ? e[0] : 0.0;
            for (int j = 0; j + 1 < n; ++j) {
                const double nd = d[j + 1] - lmb, nu = j + 2 < n ? e[j + 1] : 0.0, sub = e[j];
                if (fabs(cd) >= fabs(sub)) {
                    piv[j] = 0;
                    if (fabs(cd) < small) cd = cd >= 0.0 ? small : -small;
                    const double lj = sub / cd;
                    l[j] = lj;
                    u0i[j] = 1.0 / cd;
                    u1[j] = cu;
                    u2[j] = 0.0;
                    cd = nd - lj * cu;
                    cu = nu;
                } else {
                    piv[j] = 1;
                    const double lj = cd / sub;
                    l[j] = lj;
                    u0i[j] = 1.0 / sub;
                    u1[j] = nd;
                    u2[j] = nu;
                    cd = cu - lj * nd;
                    cu = -lj * nu;
                }
            }
            if (fabs(cd) < small) cd = cd >= 0.0 ? small : -small;
            u0i[n - 1] = 1.0 / cd;
        }
        for (int j = lane; j < n; j += 32) z[j] = hash_uniform(((uint64_t)i << 32) ^ (uint64_t)j);
        __syncwarp();
        for (int it = 0; it < 3; ++it) {
            if (lane == 0) {
                for (int j = 0; j < n; ++j) y[j] = z[j];
                for (int j = 0; j + 1 < n; ++j) {
                    if (piv[j]) {
                        const double t = y[j];
                        y[j] = y[j + 1];
                        y[j + 1] = t;
                    }
                    y[j + 1] -= l[j] * y[j];
                }
                double z1 = 0.0, z2 = 0.0;  // z[j + 1], z[j + 2]
                for (int j = n - 1; j >= 0; --j) {
                    double s = y[j];
                    if (j + 1 < n) s -= u1[j] * z1;
                    if (j + 2 < n) s -= u2[j] * z2;
                    const double zj = s * u0i[j];
                    z[j] = zj;
                    z2 = z1;
                    z1 = zj;
                }
            }
            __syncwarp();
            // orthogonal to the earlier vectors of the cluster, then unit length
            for (int jv = i0; jv < i; ++jv) {
                const double *o = Z + (size_t)jv * n;
                double s = 0.0;
                for (int j = lane; j < n; j += 32) s += o[j] * z[j];
                s = warp_sum(s);
                for (int j = lane; j < n; j += 32) z[j] -= s * o[j];
                __syncwarp();
            }
            double s = 0.0;
            for (int j = lane; j < n; j += 32) s += z[j] * z[j];
            s = warp_sum(s);
            const double inv = s > 0.0 ? 1.0 / sqrt(s) : 0.0;
            for (int j = lane; j < n; j += 32) z[j] *= inv;
            __syncwarp();
        }
    }
}

// Vectors of eigenvalues closer than kNearTol ||T||, made orthogonal in
// ascending order (one warp per chain of such neighbours).  The vector of an
// eigenvalue known to eps ||T|| carries about eps ||T|| / gap of its neighbour: a
// residual of eps ||T|| whatever the gap, 4e-7 of the neighbour at the gap of a
// cluster (below it inverse iteration), 4e-12 where this ends.
__global__ void __launch_bounds__(32) k_tri_orth(int n, int m, const double *__restrict__ bounds,
                                                 const double *__restrict__ lam, double *__restrict__ Z) {
    const int i0 = blockIdx.x, lane = threadIdx.x;
    const double tol = kNearTol * bounds[2];
    if (i0 > 0 && lam[i0] - lam[i0 - 1] <= tol) return;  // not the first of its chain
    for (int i = i0 + 1; i < m && lam[i] - lam[i - 1] <= tol; ++i) {
        double *z = Z + (size_t)i * n;
        for (int jv = i - 1; jv >= i0 && lam[i] - lam[jv] <= tol; --jv) {
            const double *o = Z + (size_t)jv * n;
            double s = 0.0;
            for (int j = lane; j < n; j += 32) s = fma(o[j], z[j], s);
            s = warp_sum(s);
            // unit length again where the part taken off is felt
            const double c = fabs(s) > 1e-9 ? rsqrt(fmax(1.0 - s * s, 0.25)) : 1.0;
            for (int j = lane; j < n; j += 32) z[j] = c * fma(-s, o[j], z[j]);
            __syncwarp();
        }
    }
}

// X[:, i] = Q z_i for i in this CTA's group; vectors kept in shared memory
__global__ void __launch_bounds__(kTriThreads) k_tri_back(int n, int m, int per_cta, const double *__restrict__ Vh,
                                                        const double *__restrict__ tau, const double *__restrict__ Z,
                                                        double *__restrict__ X, int ldx) {
    extern __shared__ double zs[];  // per_cta x n
    __shared__ double red[kTriThreads / 32][8];
    __shared__ double dots[8];
    const int i0 = blockIdx.x * per_cta;
    const int cnt = min(per_cta, m - i0);
    for (int idx = threadIdx.x; idx < cnt * n; idx += kTriThreads) zs[idx] = Z[(size_t)i0 * n + idx];
    __syncthreads();
    for (int k = n - 2; k >= 0; --k) {
        const double t = tau[k];
        if (t == 0.0) continue;  // uniform across the CTA
        const double *v = Vh + (size_t)k * n;
        double part[8];
#pragma unroll
        for (int c = 0; c < 8; ++c) part[c] = 0.0;
        for (int j = k + 1 + threadIdx.x; j < n; j += kTriThreads) {
            const double vj = v[j];
#pragma unroll
            for (int c = 0; c < 8; ++c)
                if (c < cnt) part[c] += vj * zs[c * n + j];
        }
#pragma unroll
        for (int c = 0; c < 8; ++c) {
            double s = part[c];
            for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            part[c] = s;
        }
        if ((threadIdx.x & 31) == 0)
#pragma unroll
            for (int c = 0; c < 8; ++c) red[threadIdx.x >> 5][c] = part[c];
        __syncthreads();
        if (threadIdx.x < 8) {
            double s = 0.0;
            for (int wi = 0; wi < kTriThreads / 32; ++wi) s += red[wi][threadIdx.x];
            dots[threadIdx.x] = t * s;
        }
        __syncthreads();
        for (int j = k + 1 + threadIdx.x; j < n; j += kTriThreads) {
            const double vj = v[j];
            for (int c = 0; c < cnt; ++c) zs[c * n + j] -= dots[c] * vj;
        }
        __syncthreads();
    }
    for (int idx = threadIdx.x; idx < cnt * n; idx += kTriThreads) {
        const int c = idx / n, j = idx % n;
        X[(size_t)j * ldx + i0 + c] = zs[idx];
    }
}

}  // namespace

size_t sym_eig_work_size(int n, int m) {
    // d e tau p e2 bounds(8) | Vh n^2 | Z m n | lam m | LU 5 n m (the minors' sequences before) | pivots n m bytes |
    // clusters m + 1 ints | d, e^2 in FP32 (n each) | F, 1 / F, its exponents | T of the reflector blocks
    return (size_t)5 * n + 8 + (size_t)n * n + (size_t)m * n + m + (size_t)5 * n * m + ((size_t)n * m + 7) / 8 +
           ((size_t)m + 2) / 2 + 16 + (size_t)n + 8 + (size_t)4 * n + 8 + (size_t)3 * n + 8 + (size_t)kWY * (n + kWY);
}

namespace {

// grid of k_tridiag_rows for an n x n matrix: G CTAs owning ceil(n / G) rows
// each; 0 if the rows do not fit in shared memory
int rows_grid(int n, int sms, size_t *smem, int *rmax) {
    const int G = std::max(1, std::min(sms, (n + 3) / 4));
    const int R = (n + G - 1) / G;
    *smem = ((size_t)R * n + 4 * (size_t)n) * sizeof(double);
    *rmax = R <= 4 ? 4 : R <= 8 ? 8 : 16;
    return (R <= 16 && *smem <= kTriSmemMax) ? G : 0;
}

template <int RMAX>
bool launch_tridiag_rows(cudaStream_t s, int G, size_t smem, int sms, int n, const double *A, double *d, double *e,
                         double *tau, double *Vh, double *pbuf, double *rbuf, unsigned *counter, double *err,
                         const int *amax) {
    HSIM_SMEM_LIMIT_ONCE(k_tridiag_rows<RMAX>, kTriSmemMax);
    int per_sm = 0;
    HSIM_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_tridiag_rows<RMAX>, 2 * kTrdThreads, smem));
    if ((int64_t)per_sm * sms < G) return false;
    int nn = n;
    void *args[] = {&nn, &A, &d, &e, &tau, &Vh, &pbuf, &rbuf, &counter, &err, &amax};
    HSIM_CUDA(cudaLaunchCooperativeKernel((void *)k_tridiag_rows<RMAX>, dim3(G), dim3(2 * kTrdThreads), args, smem, s));
    HSIM_LAUNCHED();
    return true;
}

template <int RPT, int NV>
void launch_back_wy(cudaStream_t s, int nv, int n, int m, const double *Vh, const double *Tw, const double *Z, double *X,
                    int ldx) {
    const size_t one = (size_t)kWY * n * sizeof(double);
    const int bufs = 2 * one <= kTriSmemMax ? 2 : 1;
    const size_t smem = bufs * one;
    HSIM_SMEM_LIMIT_ONCE((k_tri_back_wy<RPT, NV>), kTriSmemMax);
    k_tri_back_wy<RPT, NV><<<cdiv(m, nv), 128, smem, s>>>(n, m, nv, bufs, Vh, Tw, Z, X, ldx);
    HSIM_LAUNCHED();
}
template <int RPT>
void launch_back_wy(cudaStream_t s, int nv, int n, int m, const double *Vh, const double *Tw, const double *Z, double *X,
                    int ldx) {
    constexpr int kMost = RPT <= 8 ? 5 : RPT <= 12 ? 3 : 2;  // vectors that fit the registers
    nv = cdiv(nv, cdiv(nv, kMost));  // waves of equal height
    if (nv == 1) launch_back_wy<RPT, 1>(s, nv, n, m, Vh, Tw, Z, X, ldx);
    else if (nv == 2) launch_back_wy<RPT, 2>(s, nv, n, m, Vh, Tw, Z, X, ldx);
    else if (kMost > 3 && nv == 3) launch_back_wy<RPT, kMost == 5 ? 3 : 1>(s, nv, n, m, Vh, Tw, Z, X, ldx);
    else if (kMost > 4 && nv == 4) launch_back_wy<RPT, kMost == 5 ? 4 : 1>(s, nv, n, m, Vh, Tw, Z, X, ldx);
    else launch_back_wy<RPT, kMost>(s, nv, n, m, Vh, Tw, Z, X, ldx);
}

}  // namespace

void sym_eig(cudaStream_t s, int n, int m, double *A, double *evals, double *X, int ldx, double *work) {
    HSIM_CHECK_ARG(n >= 1 && m >= 1 && m <= n, "sym_eig: bad sizes");
    // p is free once T stands: the scaled diagonal
    double *d = work, *e = d + n, *tau = e + n, *p = tau + n, *ds = p, *e2 = p + n, *bounds = e2 + n;
    double *Vh = bounds + 8, *Z = Vh + (size_t)n * n, *lam = Z + (size_t)m * n, *lu = lam + m;
    unsigned char *pivf = reinterpret_cast<unsigned char *>(lu + (size_t)5 * n * m);
    int *cst = reinterpret_cast<int *>(reinterpret_cast<double *>(pivf) + ((size_t)n * m + 7) / 8);
    float *d32 = reinterpret_cast<float *>(reinterpret_cast<double *>(cst) + ((size_t)m + 2) / 2 + 8);
    float *e232 = d32 + n;
    double *pbuf = reinterpret_cast<double *>(e232 + n) + 4, *rbuf = pbuf + 2 * (size_t)n;
    double *fm = rbuf + 2 * (size_t)n, *fi = fm + n;
    int *fx = reinterpret_cast<int *>(fi + n);
    double *Tw = fi + 2 * (size_t)n;  // kWY x kWY per block of reflectors
    // sequences of k_tri_minors: 2 n m doubles, 2 ceil(n / 8) m exponents
    int *xs = reinterpret_cast<int *>(lu + (size_t)2 * n * m);
    if (n == 1) {
        HSIM_CUDA(cudaMemcpyAsync(evals, A, sizeof(double), cudaMemcpyDeviceToDevice, s));
        const double one = 1.0;
        HSIM_CUDA(cudaMemcpyAsync(X, &one, sizeof(double), cudaMemcpyHostToDevice, s));
        HSIM_CUDA(cudaStreamSynchronize(s));
        return;
    }
    int dev = 0, sms = 0;
    HSIM_CUDA(cudaGetDevice(&dev));
    HSIM_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    // HSIM_TRACE=2: stage times of every call
    static const bool detail = [] {
        const char *ev = std::getenv("HSIM_TRACE");
        return ev && std::atoi(ev) >= 2;
    }();
    cudaEvent_t t0 = nullptr, t1 = nullptr, t2 = nullptr, t3 = nullptr, t4 = nullptr;
    if (detail) {
        cudaEventCreate(&t0);
        cudaEventCreate(&t1);
        cudaEventCreate(&t2);
        cudaEventCreate(&t3);
        cudaEventCreate(&t4);
        cudaEventRecord(t0, s);
    }
    // 1. tridiagonalisation: rows resident in shared memory (one grid barrier
    // per column) where they fit, else rows in global memory (two barriers)
    size_t rsmem = 0;
    int rmax = 0;
    const int G = rows_grid(n, sms, &rsmem, &rmax);
    bool done = false;
    double *err = bounds + 4;                                       // set if a barrier gave up
    unsigned *counter = reinterpret_cast<unsigned *>(bounds + 5);  // arrivals of the barriers
    int *amax = reinterpret_cast<int *>(bounds + 6);               // largest exponent of A
    HSIM_CUDA(cudaMemsetAsync(err, 0, 3 * sizeof(double), s));
    k_symmetrize_max<<<cdiv((int64_t)n * n, kTriThreads), kTriThreads, 0, s>>>(n, A, amax);
    HSIM_LAUNCHED();
    if (G > 0) {
        if (rmax == 4) done = launch_tridiag_rows<4>(s, G, rsmem, sms, n, A, d, e, tau, Vh, pbuf, rbuf, counter, err, amax);
        else if (rmax == 8) done = launch_tridiag_rows<8>(s, G, rsmem, sms, n, A, d, e, tau, Vh, pbuf, rbuf, counter, err, amax);
        else done = launch_tridiag_rows<16>(s, G, rsmem, sms, n, A, d, e, tau, Vh, pbuf, rbuf, counter, err, amax);
    }
    const bool in_rows = done;
    if (!done) {
        const size_t smem = 2 * (size_t)n * sizeof(double);
        HSIM_CHECK_ARG(smem <= kTriSmemMax, "sym_eig: matrix too large for the tridiagonalisation kernel");
        HSIM_SMEM_LIMIT_ONCE(k_tridiag, kTriSmemMax);
        int per_sm = 0;
        HSIM_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_tridiag, kTriThreads, smem));
        HSIM_CHECK_ARG(per_sm >= 1, "sym_eig: tridiagonalisation kernel does not fit on an SM");
        const int grid = std::max(1, std::min(sms, (n + 7) / 8));
        int nn = n;
        void *args[] = {&nn, &A, &d, &e, &tau, &Vh, &p};
        HSIM_CUDA(cudaLaunchCooperativeKernel((void *)k_tridiag, dim3(grid), dim3(kTriThreads), args, smem, s));
        HSIM_LAUNCHED();
    }
    // 2. eigenvalues
    k_tri_prep<<<1, kTriThreads, 0, s>>>(n, d, e, in_rows ? amax : nullptr, ds, e2, bounds, d32, e232, fm, fi, fx);
    HSIM_LAUNCHED();
    if (detail) cudaEventRecord(t1, s);
    // about one warp per SM: G eigenvalues per warp (L = 32 / G >= 2 lanes each)
    // FP64 issues per SM sub-partition: about one warp on each of the 4 x SMs
    // sub-partitions (blocks of four warps, one per sub-partition)
    const int per_warp = std::max(1, std::min(16, (m + 4 * sms - 1) / (4 * sms)));
    const int nwarps = (m + per_warp - 1) / per_warp;
    k_tri_bisect<<<(nwarps + 3) / 4, 128, 0, s>>>(n, m, per_warp, ds, e2, d32, e232, bounds, lam);
    HSIM_LAUNCHED();
    if (detail) cudaEventRecord(t2, s);
    // 3. vectors of single eigenvalues on the device; clusters, found on the
    // host meanwhile, by inverse iteration
    k_tri_minors<<<cdiv(m, 16), 32, 0, s>>>(n, m, ds, e2, bounds, lam, lu, xs);
    HSIM_LAUNCHED();
    k_tri_vectors<<<cdiv(m, 8), 256, 0, s>>>(n, m, lu, xs, fm, fi, fx, Z);
    HSIM_LAUNCHED();
    std::vector<double> hl(m), hb(5);
    HSIM_CUDA(cudaMemcpyAsync(hl.data(), lam, m * sizeof(double), cudaMemcpyDeviceToHost, s));
    HSIM_CUDA(cudaMemcpyAsync(hb.data(), bounds, 5 * sizeof(double), cudaMemcpyDeviceToHost, s));
    HSIM_CUDA(cudaStreamSynchronize(s));
    if (hb[4] != 0.0) fail(HSIM_E_TIMEOUT, "sym_eig: a grid barrier of the tridiagonalisation gave up");
    std::vector<int> clusters;  // first, end of every cluster of two and more
    int biggest = 1;
    for (int i = 0; i < m;) {
        int j = i + 1;
        while (j < m && !(hl[j] - hl[j - 1] > kClusterTol * hb[2])) ++j;
        if (j - i > 1) {
            clusters.push_back(i);
            clusters.push_back(j);
            biggest = std::max(biggest, j - i);
        }
        i = j;
    }
    const int nclusters = (int)clusters.size() / 2;
    if (detail) cudaEventRecord(t2, s);
    if (nclusters > 0) {
        HSIM_CUDA(cudaMemcpyAsync(cst, clusters.data(), clusters.size() * sizeof(int), cudaMemcpyHostToDevice, s));
        k_tri_invit<<<nclusters, 32, 0, s>>>(n, d, e, bounds, lam, cst, Z, lu, pivf);
        HSIM_LAUNCHED();
    }
    k_tri_orth<<<m, 32, 0, s>>>(n, m, bounds, lam, Z);
    HSIM_LAUNCHED();
    if (detail) cudaEventRecord(t3, s);
    // 4. back transformation: eight reflectors at a time where a thread's rows fit
    // its registers, else one by one, a few vectors per CTA in shared memory
    if (n <= 2048) {
        k_tri_wy<<<cdiv(n - 1, kWY), 128, 0, s>>>(n, Vh, tau, Tw);
        HSIM_LAUNCHED();
        const int nv = cdiv(m, sms), rpt = cdiv(n, 128);
        if (rpt <= 1) launch_back_wy<1>(s, nv, n, m, Vh, Tw, Z, X, ldx);
        else if (rpt <= 3) launch_back_wy<3>(s, nv, n, m, Vh, Tw, Z, X, ldx);
        else if (rpt <= 6) launch_back_wy<6>(s, nv, n, m, Vh, Tw, Z, X, ldx);
        else if (rpt <= 8) launch_back_wy<8>(s, nv, n, m, Vh, Tw, Z, X, ldx);
        else if (rpt <= 12) launch_back_wy<12>(s, nv, n, m, Vh, Tw, Z, X, ldx);
        else launch_back_wy<16>(s, nv, n, m, Vh, Tw, Z, X, ldx);
    } else {
        const int per_cta = std::max(1, std::min(8, (int)(kTriSmemMax / ((size_t)n * sizeof(double)))));
        const size_t bsm = (size_t)per_cta * n * sizeof(double);
        HSIM_SMEM_LIMIT_ONCE(k_tri_back, kTriSmemMax);
        k_tri_back<<<cdiv(m, per_cta), kTriThreads, bsm, s>>>(n, m, per_cta, Vh, tau, Z, X, ldx);
        HSIM_LAUNCHED();
    }
    HSIM_CUDA(cudaMemcpyAsync(evals, lam, m * sizeof(double), cudaMemcpyDeviceToDevice, s));
    // the host vector `clusters` must outlive its copy
    if (nclusters > 0) HSIM_CUDA(cudaStreamSynchronize(s));
    if (detail) {
        cudaEventRecord(t4, s);
        cudaEventSynchronize(t4);
        float a = 0, b = 0, c = 0, dd = 0;
        cudaEventElapsedTime(&a, t0, t1);
        cudaEventElapsedTime(&b, t1, t2);
        cudaEventElapsedTime(&c, t2, t3);
        cudaEventElapsedTime(&dd, t3, t4);
        std::fprintf(stderr,
                     "[hsim] sym_eig n=%d m=%d tridiag %.2f ms eigenvalues %.2f ms vectors %.2f ms (%d clusters, "
                     "largest %d) back %.2f ms\n",
                     n, m, a, b, c, nclusters, biggest, dd);
        for (cudaEvent_t ev : {t0, t1, t2, t3, t4}) cudaEventDestroy(ev);
    }
}

}  // namespace k
}  // namespace hsim
