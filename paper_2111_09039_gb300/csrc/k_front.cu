// Multifrontal LDL^T factorisation of the shifted level matrix and its
// multi-right-hand-side solves (Alg. 1: one factorisation of S - mu M per
// level, then (S - mu M) Psi = M Phi for all q columns; Sec. 3.2 "Direct
// solver": symmetric indefinite LDL^T).
//
// Every front is a dense column-major nf x nf block of one arena; its first
// ns columns are the pivots.  Fronts of equal height in the elimination tree
// are independent and are processed by the same launches.  A front is
// factored in panels of kPanel = 32 columns (right-looking):
//   diag:    LDL^T of the 32 x 32 diagonal block (one CTA per front), written
//            back in place; FP64 fronts keep the inverse of its unit lower
//            factor there, which turns every triangle of the panel and of the
//            solves into a product (a triangle of 32 is a chain of 496
//            dependent FP64 instructions of 64 clocks and more, whatever the width);
//   panel:   L21 = A21 L11^-T D^-1;
//   update:  A22 -= L21 D L21^T on lower-triangular tiles;
// and the children's update blocks are added into the parent front
// (extend-add) before the parent is factored.  Pivoting is not used: the
// shifted Laplacian is factored as is after the fill-reducing ordering; a
// pivot below the tolerance is reported and replaced by +-tol.
//
// The solves work on row-major X (n x k, internal order) so that each row
// of a right-hand-side block is a contiguous, coalesced segment.
#include <cuda_runtime.h>

#include <algorithm>
#include <climits>
#include <type_traits>

#include "common.h"
#include "host.h"
#include "kernels.h"

namespace hsim {
namespace k {

namespace {

constexpr int P = kPanel;  // 32

__device__ __forceinline__ void tri_index(int64_t x, int &ti, int &tj) {
    // x -> (ti, tj) with ti >= tj, x = ti (ti + 1) / 2 + tj
    int t = (int)((sqrt(8.0 * (double)x + 1.0) - 1.0) * 0.5);
    while ((int64_t)t * (t + 1) / 2 > x) --t;
    while ((int64_t)(t + 1) * (t + 2) / 2 <= x) ++t;
    ti = t;
    tj = (int)(x - (int64_t)t * (t + 1) / 2);
}

template <typename T>
__global__ void k_front_assemble(int64_t nnz, const int *__restrict__ row_of, const int *__restrict__ col,
                                 const int64_t *__restrict__ dst, const double *__restrict__ S,
                                 const double *__restrict__ M, const double *__restrict__ Md, double mu,
                                 T *__restrict__ arena) {
    int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= nnz) return;
    int64_t d = dst[e];
    if (d < 0) return;
    double v = S[e];
    if (M) {
        v -= mu * M[e];
    } else {
        int r = row_of[e];
        if (r == col[e]) v -= mu * Md[r];
    }
    arena[d] = (T)v;
}

// extend-add of the update blocks of `children` into their parents
template <typename T>
__global__ void k_extend_add(FrontDev fd, const int *__restrict__ parent, const int *__restrict__ children,
                             T *__restrict__ arena) {
    const int c = children[blockIdx.x];
    const int nsc = fd.ns[c], nfc = fd.nf[c];
    const int u = nfc - nsc;
    const int nt = (u + 31) / 32;
    int ti, tj;
    tri_index(blockIdx.y, ti, tj);
    if (ti >= nt) return;
    const int p = parent[c];
    const int nfp = fd.nf[p];
    const int *rel = fd.relmap + fd.relmap_off[c];
    const T *Fc = arena + fd.foff[c];
    T *Fp = arena + fd.foff[p];
    const int jl = threadIdx.x & 31;
    const int j = tj * 32 + jl;
    if (j >= u) return;
    const int pj = rel[j];
    for (int il = threadIdx.x >> 5; il < 32; il += blockDim.x >> 5) {
        int i = ti * 32 + il;
        if (i >= u || i < j) continue;
        T v = Fc[(int64_t)(nsc + j) * nfc + (nsc + i)];
        if (v != T(0)) atomicAdd(&Fp[(int64_t)pj * nfp + rel[i]], v);
    }
}

// Factor the kb x kb diagonal block held in smem column-major D[c][r]
// (LDL^T, unit L below the diagonal, D on the diagonal).
template <typename T>
__device__ void ldlt_block(T (*Dg)[P + 1], int kb, double tol, int *flags) {
    __shared__ T lj[P];
    for (int j = 0; j < kb; ++j) {
        __syncthreads();
        T d = Dg[j][j];
        if (!(fabs((double)d) >= tol)) {  // also catches NaN
            if (threadIdx.x == 0) atomicAdd(&flags[0], 1);
            d = (d < T(0)) ? (T)-tol : (T)tol;
        }
        for (int i = j + 1 + threadIdx.x; i < kb; i += blockDim.x) lj[i] = Dg[j][i] / d;
        __syncthreads();
        for (int idx = threadIdx.x; idx < (kb - j - 1) * (kb - j - 1); idx += blockDim.x) {
            int r = j + 1 + idx % (kb - j - 1);
            int c = j + 1 + idx / (kb - j - 1);
            if (r >= c) Dg[c][r] -= lj[r] * d * lj[c];
        }
        __syncthreads();
        if (threadIdx.x == 0) Dg[j][j] = d;
        for (int i = j + 1 + threadIdx.x; i < kb; i += blockDim.x) Dg[j][i] = lj[i];
    }
    __syncthreads();
}

constexpr int kPanelRows = 128;

// LDL^T of the kb x kb diagonal block of panel k0, one CTA per front,
// written back in place (unit L below the diagonal, D on it).
template <typename T>
__global__ void __launch_bounds__(128) k_front_diag_block(FrontDev fd, const int *__restrict__ nodes, int k0,
                                                          T *__restrict__ arena, double tol, int *flags) {
    __shared__ T Dg[P][P + 1];
    const int t = nodes[blockIdx.x];
    const int nf = fd.nf[t], ns = fd.ns[t];
    const int kb = min(P, ns - k0);
    if (kb <= 0) return;
    T *F = arena + fd.foff[t];
    for (int idx = threadIdx.x; idx < kb * kb; idx += blockDim.x) {
        int r = idx % kb, c = idx / kb;
        Dg[c][r] = (r >= c) ? F[(int64_t)(k0 + c) * nf + (k0 + r)] : 0.0;
    }
    ldlt_block(Dg, kb, tol, flags);
    for (int idx = threadIdx.x; idx < kb * kb; idx += blockDim.x) {
        int r = idx % kb, c = idx / kb;
        if (r >= c) F[(int64_t)(k0 + c) * nf + (k0 + r)] = Dg[c][r];
    }
}

// Rows below the diagonal block: x L11^T = a, l = x / d, with L11 and D
// read from the block factored by k_front_diag_block in the previous launch.
template <typename T>
__global__ void __launch_bounds__(128) k_front_panel(FrontDev fd, const int *__restrict__ nodes, int k0,
                                                     T *__restrict__ arena) {
    __shared__ T Dg[P][P + 1];
    const int t = nodes[blockIdx.x];
    const int nf = fd.nf[t], ns = fd.ns[t];
    const int kb = min(P, ns - k0);
    if (kb <= 0) return;
    const int r0 = k0 + kb + blockIdx.y * kPanelRows;
    if (r0 >= nf) return;
    T *F = arena + fd.foff[t];
    for (int idx = threadIdx.x; idx < kb * kb; idx += blockDim.x) {
        int r = idx % kb, c = idx / kb;
        Dg[c][r] = (r >= c) ? F[(int64_t)(k0 + c) * nf + (k0 + r)] : 0.0;
    }
    __syncthreads();
    const int r = r0 + threadIdx.x;
    if (r < nf) {
        T x[P];
#pragma unroll
        for (int c = 0; c < P; ++c)
            if (c < kb) x[c] = F[(int64_t)(k0 + c) * nf + r];
#pragma unroll
        for (int c = 0; c < P; ++c) {
            if (c < kb) {
                T v = x[c];
#pragma unroll
                for (int cc = 0; cc < P; ++cc)
                    if (cc < c) v -= x[cc] * Dg[cc][c];
                x[c] = v;
            }
        }
#pragma unroll
        for (int c = 0; c < P; ++c)
            if (c < kb) F[(int64_t)(k0 + c) * nf + r] = x[c] / Dg[c][c];
    }
}

// FP64 diagonal block: D and the inverse of L11 in one pass (Gauss-Jordan on [A |
// I] without the part above the diagonal).  Lane r of every warp holds row r,
// warp w the columns w, w + 4, ... of the block and of the inverse, so a pivot
// step is up to 8 + 8 FP64 instructions per warp, one warp per SM sub-partition,
// around a chain of reciprocal, product and update.  32 pivots take 28 us;
// with the block in shared memory, three barriers a pivot and a division per
// entry they took 36.6, without the inverse.  (A correction step on the quotients
// of l and of the panel left the solves' error as it was.)
__global__ void __launch_bounds__(128) k_front_diag_inv(FrontDev fd, const int *__restrict__ nodes, int k0,
                                                        double *__restrict__ arena, double tol, int *flags) {
    __shared__ double u[2][P], pinv[2];
    const int t = nodes[blockIdx.x];
    const int nf = fd.nf[t], ns = fd.ns[t];
    const int kb = min(P, ns - k0);
    if (kb <= 0) return;
    const int r = threadIdx.x & 31, w = threadIdx.x >> 5;
    double *F = arena + fd.foff[t] + (int64_t)k0 * nf + k0;  // column c at F + c nf
    double a[P / 4], e[P / 4];
#pragma unroll
    for (int q = 0; q < P / 4; ++q) {
        const int c = w + 4 * q;
        a[q] = c < kb && r < kb && r >= c ? F[(int64_t)c * nf + r] : 0.0;
        e[q] = r == c ? 1.0 : 0.0;
    }
#pragma unroll
    for (int j = 0; j < P; ++j) {
        if (j >= kb) break;
        if (w == (j & 3)) {
            double d = __shfl_sync(0xffffffffu, a[j / 4], j);
            if (!(fabs(d) >= tol)) {  // also catches NaN
                if (r == 0) atomicAdd(&flags[0], 1);
                d = d < 0.0 ? -tol : tol;
                if (r == j) a[j / 4] = d;
            }
            u[j & 1][r] = a[j / 4];
            if (r == 0) pinv[j & 1] = 1.0 / d;
        }
        __syncthreads();
        // row r > j: l = a_rj / d, A_r -= l (d l_c) = l u_c, I_r -= l I_j
        const double l = r > j ? u[j & 1][r] * pinv[j & 1] : 0.0;
#pragma unroll
        for (int q = 0; q < P / 4; ++q) {
            const int c = w + 4 * q;
            if (c > j) a[q] = fma(-l, u[j & 1][c], a[q]);
        }
#pragma unroll
        for (int q = 0; q < P / 4; ++q)
            if (4 * q <= j) e[q] = fma(-l, __shfl_sync(0xffffffffu, e[q], j), e[q]);
    }
#pragma unroll
    for (int q = 0; q < P / 4; ++q) {
        const int c = w + 4 * q;
        if (c < kb && r < kb && r >= c) F[(int64_t)c * nf + r] = r == c ? a[q] : e[q];
    }
}

// FP64 rows below the diagonal block: L21 = A21 Linv^T D^-1 with the inverse that
// k_front_diag_inv left in the block.  A CTA takes 16 rows, thread (row, column
// group g) the columns g, g + 8, g + 16, g + 24: small tiles, since the FP64
// pipes of idle SMs are what a panel of a few hundred rows can use.
constexpr int kPanelRows64 = 16;
__global__ void __launch_bounds__(128) k_front_panel64(FrontDev fd, const int *__restrict__ nodes, int k0,
                                                       double *__restrict__ arena) {
    __shared__ double Li[P][P + 1], As[P][kPanelRows64 + 1], di[P];
    const int t = nodes[blockIdx.x];
    const int nf = fd.nf[t], ns = fd.ns[t];
    const int kb = min(P, ns - k0);
    if (kb <= 0) return;
    const int r0 = k0 + kb + blockIdx.y * kPanelRows64;
    if (r0 >= nf) return;
    double *F = arena + fd.foff[t];
    for (int idx = threadIdx.x; idx < P * P; idx += 128) {
        const int r = idx & 31, c = idx >> 5;
        Li[r][c] = r > c && r < kb ? F[(int64_t)(k0 + c) * nf + (k0 + r)] : r == c ? 1.0 : 0.0;
    }
    for (int idx = threadIdx.x; idx < P * kPanelRows64; idx += 128) {
        const int r = idx % kPanelRows64, c = idx / kPanelRows64;
        As[c][r] = c < kb && r0 + r < nf ? F[(int64_t)(k0 + c) * nf + (r0 + r)] : 0.0;
    }
    if (threadIdx.x < kb) di[threadIdx.x] = 1.0 / F[(int64_t)(k0 + threadIdx.x) * nf + (k0 + threadIdx.x)];
    __syncthreads();
    const int r = threadIdx.x % kPanelRows64, g = threadIdx.x / kPanelRows64;
    double acc[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll
    for (int v = 0; v < 4; ++v)
        // the upper part is zero: whole groups of eight columns up to this one
        for (int cc = 0; cc < 8 * v + 8; ++cc) acc[v] = fma(As[cc][r], Li[g + 8 * v][cc], acc[v]);
#pragma unroll
    for (int v = 0; v < 4; ++v) {
        const int c = g + 8 * v;
        if (c < kb && r0 + r < nf) F[(int64_t)(k0 + c) * nf + (r0 + r)] = acc[v] * di[c];
    }
}

// A22 -= L21 D L21^T on TS x TS lower-triangular tiles of the trailing block;
// with ntj > 0 only the columns below c_end (tile y = ti * ntj + tj)
template <typename T, int TS>
__global__ void __launch_bounds__(256) k_front_update(FrontDev fd, const int *__restrict__ nodes, int k0,
                                                      T *__restrict__ arena, int c_end, int ntj) {
    __shared__ T Lr[P][TS];
    __shared__ T Lc[P][TS];
    const int t = nodes[blockIdx.x];
    const int nf = fd.nf[t], ns = fd.ns[t];
    const int kb = min(P, ns - k0);
    if (kb <= 0) return;
    const int base = k0 + kb;
    const int m = nf - base;
    if (m <= 0) return;
    const int nt = (m + TS - 1) / TS;
    int ti, tj;
    if (ntj > 0) {
        ti = (int)(blockIdx.y / ntj);
        tj = (int)(blockIdx.y % ntj);
        if (ti < tj) return;
    } else {
        tri_index(blockIdx.y, ti, tj);
    }
    if (ti >= nt) return;
    T *F = arena + fd.foff[t];
    const int r0 = base + ti * TS, c0 = base + tj * TS;
    if (c0 >= c_end) return;
    for (int idx = threadIdx.x; idx < P * TS; idx += blockDim.x) {
        int i = idx % TS, kk = idx / TS;
        T vr = 0.0, vc = 0.0;
        if (kk < kb) {
            T d = F[(int64_t)(k0 + kk) * nf + (k0 + kk)];
            if (r0 + i < nf) vr = F[(int64_t)(k0 + kk) * nf + (r0 + i)];
            if (c0 + i < nf) vc = F[(int64_t)(k0 + kk) * nf + (c0 + i)] * d;
        }
        Lr[kk][i] = vr;
        Lc[kk][i] = vc;
    }
    __syncthreads();
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    constexpr int U = TS / 16;
    T acc[U][U] = {};
    for (int kk = 0; kk < kb; ++kk) {
        T a[U], b[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            a[u] = Lr[kk][ty + 16 * u];
            b[u] = Lc[kk][tx + 16 * u];
        }
#pragma unroll
        for (int u = 0; u < U; ++u)
#pragma unroll
            for (int v = 0; v < U; ++v) acc[u][v] += a[u] * b[v];
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
        int r = r0 + ty + 16 * u;
        if (r >= nf) continue;
#pragma unroll
        for (int v = 0; v < U; ++v) {
            int c = c0 + tx + 16 * v;
            if (c < nf && r >= c && c < c_end) F[(int64_t)c * nf + r] -= acc[u][v];
        }
    }
}

template <typename T>
__global__ void k_front_diag(FrontDev fd, const int *__restrict__ nodes, int n_nodes,
                             const T *__restrict__ arena, T *__restrict__ dpos, int *neg) {
    int t_idx = blockIdx.x;
    if (t_idx >= n_nodes) return;
    int t = nodes[t_idx];
    const int nf = fd.nf[t], ns = fd.ns[t], ps = fd.pstart[t];
    const T *F = arena + fd.foff[t];
    int cnt = 0;
    for (int i = threadIdx.x; i < ns; i += blockDim.x) {
        T d = F[(int64_t)i * nf + i];
        dpos[ps + i] = d;
        cnt += (d < T(0));
    }
    if (cnt) atomicAdd(neg, cnt);
}

template <typename T>
__global__ void k_front_maxdiag(FrontDev fd, const T *__restrict__ arena, unsigned long long *out) {
    const int t = blockIdx.x;
    const int nf = fd.nf[t], ns = fd.ns[t];
    const T *F = arena + fd.foff[t];
    unsigned long long best = 0;
    for (int i = threadIdx.x; i < ns; i += blockDim.x) {
        unsigned long long b = (unsigned long long)__double_as_longlong(fabs((double)F[(int64_t)i * nf + i]));
        best = b > best ? b : best;
    }
    if (best) atomicMax(out, best);
}

// ---- FP64 solves (FP32 factors are solved in the inverted form, k_finv.cu) -----
// Every diagonal block holds the inverse of its unit lower factor (k_front_diag_inv),
// so the triangles are products; tiles are small where a height has few fronts
// (an SM's FP64 pipes take 1.7 to 1.9 lanes per clock: 64 x 64 x 32 products keep one
// SM busy for 38 us while others idle).

// Li[r][c] = the inverse block (rows and columns beyond kb: identity)
__device__ __forceinline__ void load_inv(double (&Li)[P][P + 1], const double *__restrict__ F, int nf, int k0, int kb) {
    for (int idx = threadIdx.x; idx < P * P; idx += blockDim.x) {
        const int r = idx & 31, c = idx >> 5;
        Li[r][c] = r > c && r < kb ? F[(int64_t)(k0 + c) * nf + (k0 + r)] : r == c ? 1.0 : 0.0;
    }
}

constexpr int kTriCols = 16;

// X[panel rows, cols] = Linv X[...] (backward: Linv^T X[...]); thread (column,
// row group g): rows g, g + 8, g + 16, g + 24 of a 16-column tile
template <bool TRANS>
__global__ void __launch_bounds__(128) k_solve_tri(FrontDev fd, const int *__restrict__ nodes, int k0,
                                                   const double *__restrict__ arena, int k, double *__restrict__ X,
                                                   int ldx) {
    __shared__ double Li[P][P + 1], Xs[P][kTriCols];
    const int t = nodes[blockIdx.x];
    const int nf = fd.nf[t], ns = fd.ns[t], ps = fd.pstart[t];
    const int kb = min(P, ns - k0);
    if (kb <= 0) return;
    load_inv(Li, arena + fd.foff[t], nf, k0, kb);
    const int c = threadIdx.x % kTriCols, g = threadIdx.x / kTriCols, j = blockIdx.y * kTriCols + c;
    double *Xb = X + (size_t)(ps + k0) * ldx + j;
#pragma unroll
    for (int v = 0; v < 4; ++v) {
        const int r = g + 8 * v;
        Xs[r][c] = r < kb && j < k ? Xb[(size_t)r * ldx] : 0.0;
    }
    __syncthreads();
    double acc[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll
    for (int v = 0; v < 4; ++v) {
        const int r = g + 8 * v;
        if (TRANS) {
            for (int q = 8 * v; q < P; ++q) acc[v] = fma(Li[q][r], Xs[q][c], acc[v]);
        } else {
            for (int q = 0; q < 8 * v + 8; ++q) acc[v] = fma(Li[r][q], Xs[q][c], acc[v]);
        }
    }
    if (j >= k) return;
#pragma unroll
    for (int v = 0; v < 4; ++v) {
        const int r = g + 8 * v;
        if (r < kb) Xb[(size_t)r * ldx] = acc[v];
    }
}

// X[row(r), cols] -= sum_c L[r, k0+c] X[panel row c, cols] for front rows
// r >= k0 + kb on TS x TS tiles; pivot rows of the front are updated in place,
// rows of ancestor fronts with atomics (sibling fronts share them).
template <int TS>
__global__ void __launch_bounds__(256) k_solve_fwd_upd(FrontDev fd, const int *__restrict__ nodes, int k0,
                                                       const double *__restrict__ arena, int k,
                                                       double *__restrict__ X, int ldx) {
    constexpr int U = TS / 16;
    __shared__ double Ls[P][TS];
    __shared__ double Xs[P][TS];
    const int t = nodes[blockIdx.x];
    const int nf = fd.nf[t], ns = fd.ns[t], ps = fd.pstart[t];
    const int kb = min(P, ns - k0);
    if (kb <= 0) return;
    const int r0 = k0 + kb + blockIdx.y * TS;
    if (r0 >= nf) return;
    const int c0 = blockIdx.z * TS;
    if (c0 >= k) return;
    const double *F = arena + fd.foff[t];
    const int *rows = fd.rows + fd.rows_off[t];
    for (int idx = threadIdx.x; idx < P * TS; idx += blockDim.x) {
        const int i = idx % TS, kk = idx / TS;
        double lv = 0.0, xv = 0.0;
        if (kk < kb) {
            if (r0 + i < nf) lv = F[(int64_t)(k0 + kk) * nf + (r0 + i)];
            if (c0 + i < k) xv = X[(size_t)(ps + k0 + kk) * ldx + c0 + i];
        }
        Ls[kk][i] = lv;
        Xs[kk][i] = xv;
    }
    __syncthreads();
    // thread: rows ty + 16 u, U contiguous columns
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    double acc[U][U] = {};
    for (int kk = 0; kk < kb; ++kk) {
        double a[U], b[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            a[u] = Ls[kk][ty + 16 * u];
            b[u] = Xs[kk][U * tx + u];
        }
#pragma unroll
        for (int u = 0; u < U; ++u)
#pragma unroll
            for (int v = 0; v < U; ++v) acc[u][v] = fma(a[u], b[v], acc[u][v]);
    }
    const int cb = c0 + U * tx;
#pragma unroll
    for (int u = 0; u < U; ++u) {
        const int r = r0 + ty + 16 * u;
        if (r >= nf) continue;
        double *xr = X + (size_t)rows[r] * ldx + cb;
#pragma unroll
        for (int v = 0; v < U; ++v) {
            if (cb + v >= k) break;
            if (r < ns) xr[v] -= acc[u][v];
            else atomicAdd(xr + v, -acc[u][v]);
        }
    }
}

__global__ void k_solve_diag(int n, int k, const double *__restrict__ dpos, double *__restrict__ X, int ldx) {
    int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (int64_t)n * k) return;
    int i = (int)(idx / k), j = (int)(idx % k);
    X[(size_t)i * ldx + j] /= dpos[i];
}

// X[panel rows c, cols] -= sum_{r >= k0+kb} L[r, k0+c] X[row(r), cols].  A CTA
// covers one 32-row chunk of r and CT columns; when one CTA covers all rows of
// the front (grid.y == 1) it updates the panel rows with plain stores, otherwise
// the partial sums are accumulated with atomics.
template <int CT>
__global__ void __launch_bounds__(256) k_solve_bwd_upd(FrontDev fd, const int *__restrict__ nodes, int k0,
                                                       const double *__restrict__ arena, int k,
                                                       double *__restrict__ X, int ldx) {
    constexpr int RS = 256 / CT, NU = P / RS;  // panel rows cb, cb + RS, ... per thread
    __shared__ double Ls[P][P + 1];  // [r][c]
    __shared__ double Xs[P][CT];     // [r][col]
    const int t = nodes[blockIdx.x];
    const int nf = fd.nf[t], ns = fd.ns[t], ps = fd.pstart[t];
    const int kb = min(P, ns - k0);
    if (kb <= 0) return;
    const int r0 = k0 + kb + blockIdx.y * P;
    if (r0 >= nf) return;
    const int c0 = blockIdx.z * CT;
    if (c0 >= k) return;
    const double *F = arena + fd.foff[t];
    const int *rows = fd.rows + fd.rows_off[t];
    for (int idx = threadIdx.x; idx < P * P; idx += 256) {
        const int r = idx % P, c = idx / P;
        Ls[r][c] = (r0 + r < nf && c < kb) ? F[(int64_t)(k0 + c) * nf + (r0 + r)] : 0.0;
    }
    for (int idx = threadIdx.x; idx < P * CT; idx += 256) {
        const int jj = idx % CT, r = idx / CT;
        Xs[r][jj] = (r0 + r < nf && c0 + jj < k) ? X[(size_t)rows[r0 + r] * ldx + c0 + jj] : 0.0;
    }
    __syncthreads();
    const int j = threadIdx.x % CT, cb = threadIdx.x / CT;
    double acc[NU] = {};
    for (int r = 0; r < min(P, nf - r0); ++r) {
        const double xv = Xs[r][j];
#pragma unroll
        for (int u = 0; u < NU; ++u) acc[u] = fma(Ls[r][cb + RS * u], xv, acc[u]);
    }
    if (c0 + j < k) {
        const bool whole = gridDim.y == 1;
#pragma unroll
        for (int u = 0; u < NU; ++u) {
            const int c = cb + RS * u;
            if (c < kb) {
                double *x = &X[(size_t)(ps + k0 + c) * ldx + c0 + j];
                if (whole) *x -= acc[u];
                else atomicAdd(x, -acc[u]);
            }
        }
    }
}

// ---- single-panel fronts (ns <= P, nf <= kSmallNf): fused solve kernels -------
// One CTA per (front, column tile): the front's L panel and pivot rows are
// staged in shared memory once; the forward kernel multiplies the pivot rows by
// Linv and sends L21 x1 to the ancestors' rows (atomics), the backward kernel
// gathers the ancestors' rows, subtracts L21^T x2 and multiplies by Linv^T.
// Thread layout: SC columns x 256 / SC row groups.
template <int SC>
__global__ void __launch_bounds__(256) k_solve_fwd_small(FrontDev fd, const int *__restrict__ nodes,
                                                         const double *__restrict__ arena, int k,
                                                         double *__restrict__ X, int ldx, int nf_max) {
    constexpr int RG = 256 / SC;
    extern __shared__ __align__(16) unsigned char small_smem[];
    double *Ls = reinterpret_cast<double *>(small_smem);  // ns x nf (column-major panel)
    double *Xp = Ls + P * nf_max, *Yp = Xp + P * SC;       // [P][SC] each
    const int t = nodes[blockIdx.x];
    const int nf = fd.nf[t], ns = fd.ns[t], ps = fd.pstart[t];
    const int c0 = blockIdx.y * SC;
    if (c0 >= k) return;
    const int tid = threadIdx.x, c = tid % SC, rg = tid / SC;
    const bool live = c0 + c < k;
    const double *F = arena + fd.foff[t];
    for (int i = tid; i < ns * nf; i += 256) Ls[i] = F[i];
    double *Xc = X + c0 + c;
    for (int r = rg; r < ns; r += RG) Xp[r * SC + c] = live ? Xc[(size_t)(ps + r) * ldx] : 0.0;
    __syncthreads();
    for (int r = rg; r < ns; r += RG) {
        double acc = Xp[r * SC + c];
        for (int q = 0; q < r; ++q) acc = fma(Ls[q * nf + r], Xp[q * SC + c], acc);
        Yp[r * SC + c] = acc;
        if (live) Xc[(size_t)(ps + r) * ldx] = acc;
    }
    __syncthreads();
    // ancestors' rows: x_r -= L_r. x_p, two rows at a time
    const int *rows = fd.rows + fd.rows_off[t];
    for (int r = ns + rg; r < nf; r += 2 * RG) {
        const int r2 = r + RG < nf ? r + RG : r;
        double a0 = 0.0, a1 = 0.0;
        for (int q = 0; q < ns; ++q) {
            const double y = Yp[q * SC + c];
            a0 = fma(Ls[q * nf + r], y, a0);
            a1 = fma(Ls[q * nf + r2], y, a1);
        }
        if (live) {
            atomicAdd(Xc + (size_t)rows[r] * ldx, -a0);
            if (r2 != r) atomicAdd(Xc + (size_t)rows[r2] * ldx, -a1);
        }
    }
}

template <int SC>
__global__ void __launch_bounds__(256) k_solve_bwd_small(FrontDev fd, const int *__restrict__ nodes,
                                                         const double *__restrict__ arena, int k,
                                                         double *__restrict__ X, int ldx, int nf_max) {
    constexpr int RG = 256 / SC;
    extern __shared__ __align__(16) unsigned char small_smem[];
    double *Ls = reinterpret_cast<double *>(small_smem);
    double *Xp = Ls + P * nf_max;    // [P][SC]
    double *Xu = Xp + P * SC;        // [P][SC] chunk of ancestor rows
    const int t = nodes[blockIdx.x];
    const int nf = fd.nf[t], ns = fd.ns[t], ps = fd.pstart[t];
    const int c0 = blockIdx.y * SC;
    if (c0 >= k) return;
    const int tid = threadIdx.x, c = tid % SC, rg = tid / SC;
    const bool live = c0 + c < k;
    const double *F = arena + fd.foff[t];
    const int *rows = fd.rows + fd.rows_off[t];
    for (int i = tid; i < ns * nf; i += 256) Ls[i] = F[i];
    double *Xc = X + c0 + c;
    // x_p - L21^T x_u over 32-row chunks of the ancestors' rows; thread: pivots
    // q = rg + RG j of its column
    constexpr int QJ = (P + RG - 1) / RG;
    double acc[QJ];
#pragma unroll
    for (int j = 0; j < QJ; ++j) {
        const int q = rg + RG * j;
        acc[j] = q < ns && live ? Xc[(size_t)(ps + q) * ldx] : 0.0;
    }
    for (int r0 = ns; r0 < nf; r0 += P) {
        const int cnt = min(P, nf - r0);
        __syncthreads();
        for (int rr = rg; rr < cnt; rr += RG) Xu[rr * SC + c] = live ? Xc[(size_t)rows[r0 + rr] * ldx] : 0.0;
        __syncthreads();
        for (int rr = 0; rr < cnt; ++rr) {
            const double xu = -Xu[rr * SC + c];
#pragma unroll
            for (int j = 0; j < QJ; ++j) {
                const int q = rg + RG * j;
                if (q < ns) acc[j] = fma(Ls[q * nf + r0 + rr], xu, acc[j]);
            }
        }
    }
#pragma unroll
    for (int j = 0; j < QJ; ++j) {
        const int q = rg + RG * j;
        if (q < ns) Xp[q * SC + c] = acc[j];
    }
    __syncthreads();
    for (int r = rg; r < ns; r += RG) {
        double a = Xp[r * SC + c];
        for (int q = r + 1; q < ns; ++q) a = fma(Ls[r * nf + q], Xp[q * SC + c], a);
        if (live) Xc[(size_t)(ps + r) * ldx] = a;
    }
}

inline unsigned cdiv(int64_t a, int64_t b) { return (unsigned)((a + b - 1) / b); }

}  // namespace

template <typename T>
void front_assemble(cudaStream_t s, int64_t nnz, const int *row_of, const int *col, const int64_t *dst,
                    const double *S_val, const double *M_val, const double *M_diag, double mu, T *arena) {
    if (nnz <= 0) return;
    k_front_assemble<T><<<cdiv(nnz, 256), 256, 0, s>>>(nnz, row_of, col, dst, S_val, M_val, M_diag, mu, arena);
    HSIM_LAUNCHED();
}

template <typename T>
void front_extend_add(cudaStream_t s, const FrontDev &fd, const int *parent, const int *children, int n_children,
                      int max_upd, T *arena) {
    if (n_children <= 0 || max_upd <= 0) return;
    int64_t Tt = (max_upd + 31) / 32;
    dim3 g((unsigned)n_children, (unsigned)(Tt * (Tt + 1) / 2));
    k_extend_add<T><<<g, 256, 0, s>>>(fd, parent, children, arena);
    HSIM_LAUNCHED();
}

static int front_sms() {
    int dev = 0, c = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&c, cudaDevAttrMultiProcessorCount, dev);
    return c > 0 ? c : 1;
}

template <typename T>
void front_panel(cudaStream_t s, const FrontDev &fd, const int *nodes, int n_nodes, int k0, int max_rows, T *arena,
                 double pivot_tol, int *flags) {
    if (n_nodes <= 0) return;
    if constexpr (std::is_same<T, double>::value) {
        k_front_diag_inv<<<(unsigned)n_nodes, 128, 0, s>>>(fd, nodes, k0, arena, pivot_tol, flags);
        HSIM_LAUNCHED();
        if (max_rows <= 0) return;
        dim3 g((unsigned)n_nodes, cdiv(max_rows, kPanelRows64));
        k_front_panel64<<<g, 128, 0, s>>>(fd, nodes, k0, arena);
        HSIM_LAUNCHED();
    } else {
        k_front_diag_block<T><<<(unsigned)n_nodes, 128, 0, s>>>(fd, nodes, k0, arena, pivot_tol, flags);
        HSIM_LAUNCHED();
        if (max_rows <= 0) return;
        dim3 g((unsigned)n_nodes, cdiv(max_rows, kPanelRows));
        k_front_panel<T><<<g, 128, 0, s>>>(fd, nodes, k0, arena);
        HSIM_LAUNCHED();
    }
}

template <typename T, int TS>
static void launch_update(cudaStream_t s, const FrontDev &fd, const int *nodes, int n_nodes, int k0, int max_trail,
                          T *arena, int c_end) {
    int64_t Tt = (max_trail + TS - 1) / TS;
    // column tiles below c_end (the trailing part starts after k0's first pivot)
    const int64_t ntj = c_end == INT_MAX ? 0 : std::min<int64_t>(Tt, (c_end - k0 + TS - 2) / TS + 1);
    if (c_end != INT_MAX && ntj <= 0) return;
    dim3 g((unsigned)n_nodes, (unsigned)(ntj > 0 ? Tt * ntj : Tt * (Tt + 1) / 2));
    k_front_update<T, TS><<<g, 256, 0, s>>>(fd, nodes, k0, arena, c_end, (int)ntj);
    HSIM_LAUNCHED();
}

template <typename T>
void front_update(cudaStream_t s, const FrontDev &fd, const int *nodes, int n_nodes, int k0, int max_trail, T *arena,
                  int c_end) {
    if (n_nodes <= 0 || max_trail <= 0) return;
    if constexpr (std::is_same<T, double>::value) {
        // tiles of 64 keep an SM's FP64 pipes busy for 38 us, of 32 for 10, of 16
        // for 2.4: the largest with two CTAs per SM
        auto ctas = [&](int ts) {
            const int64_t q = (max_trail + ts - 1) / ts;
            return (int64_t)n_nodes * q * (q + 1) / 2;
        };
        const int64_t want = 2 * (int64_t)front_sms();
        if (ctas(64) >= want) launch_update<T, 64>(s, fd, nodes, n_nodes, k0, max_trail, arena, c_end);
        else if (ctas(32) >= want) launch_update<T, 32>(s, fd, nodes, n_nodes, k0, max_trail, arena, c_end);
        else launch_update<T, 16>(s, fd, nodes, n_nodes, k0, max_trail, arena, c_end);
    } else {
        launch_update<T, 64>(s, fd, nodes, n_nodes, k0, max_trail, arena, c_end);
    }
}

template <typename T>
void front_maxdiag(cudaStream_t s, const FrontDev &fd, int n_nodes, const T *arena, unsigned long long *out) {
    if (n_nodes <= 0) return;
    k_front_maxdiag<T><<<n_nodes, 128, 0, s>>>(fd, arena, out);
    HSIM_LAUNCHED();
}

template <typename T>
void front_diag(cudaStream_t s, const FrontDev &fd, const int *nodes, int n_nodes, const T *arena, T *dpos,
                int *neg_count) {
    if (n_nodes <= 0) return;
    k_front_diag<T><<<n_nodes, 128, 0, s>>>(fd, nodes, n_nodes, arena, dpos, neg_count);
    HSIM_LAUNCHED();
}

void solve_fwd_tri(cudaStream_t s, const FrontDev &fd, const int *nodes, int n_nodes, int k0, const double *arena,
                   int k, double *X, int ldx) {
    if (n_nodes <= 0 || k <= 0) return;
    dim3 g((unsigned)n_nodes, cdiv(k, kTriCols));
    k_solve_tri<false><<<g, 128, 0, s>>>(fd, nodes, k0, arena, k, X, ldx);
    HSIM_LAUNCHED();
}

void solve_fwd_upd(cudaStream_t s, const FrontDev &fd, const int *nodes, int n_nodes, int k0, int max_rows,
                   const double *arena, int k, double *X, int ldx) {
    if (n_nodes <= 0 || k <= 0 || max_rows <= 0) return;
    // the largest tile with two CTAs per SM (as front_update)
    auto grid = [&](int ts) { return dim3((unsigned)n_nodes, cdiv(max_rows, ts), cdiv(k, ts)); };
    auto ctas = [&](int ts) { return (int64_t)n_nodes * cdiv(max_rows, ts) * cdiv(k, ts); };
    const int64_t want = 2 * (int64_t)front_sms();
    if (ctas(64) >= want) k_solve_fwd_upd<64><<<grid(64), 256, 0, s>>>(fd, nodes, k0, arena, k, X, ldx);
    else if (ctas(32) >= want) k_solve_fwd_upd<32><<<grid(32), 256, 0, s>>>(fd, nodes, k0, arena, k, X, ldx);
    else k_solve_fwd_upd<16><<<grid(16), 256, 0, s>>>(fd, nodes, k0, arena, k, X, ldx);
    HSIM_LAUNCHED();
}

void solve_diag(cudaStream_t s, int n, int k, const double *dpos, double *X, int ldx) {
    if (n <= 0 || k <= 0) return;
    k_solve_diag<<<cdiv((int64_t)n * k, 256), 256, 0, s>>>(n, k, dpos, X, ldx);
    HSIM_LAUNCHED();
}

void solve_bwd_upd(cudaStream_t s, const FrontDev &fd, const int *nodes, int n_nodes, int k0, int max_rows,
                   const double *arena, int k, double *X, int ldx) {
    if (n_nodes <= 0 || k <= 0 || max_rows <= 0) return;
    auto grid = [&](int ct) { return dim3((unsigned)n_nodes, cdiv(max_rows, P), cdiv(k, ct)); };
    if ((int64_t)n_nodes * cdiv(max_rows, P) * cdiv(k, 64) >= 2 * (int64_t)front_sms())
        k_solve_bwd_upd<64><<<grid(64), 256, 0, s>>>(fd, nodes, k0, arena, k, X, ldx);
    else
        k_solve_bwd_upd<16><<<grid(16), 256, 0, s>>>(fd, nodes, k0, arena, k, X, ldx);
    HSIM_LAUNCHED();
}

void solve_bwd_tri(cudaStream_t s, const FrontDev &fd, const int *nodes, int n_nodes, int k0, const double *arena,
                   int k, double *X, int ldx) {
    if (n_nodes <= 0 || k <= 0) return;
    dim3 g((unsigned)n_nodes, cdiv(k, kTriCols));
    k_solve_tri<true><<<g, 128, 0, s>>>(fd, nodes, k0, arena, k, X, ldx);
    HSIM_LAUNCHED();
}

constexpr int kSmallCols = 32;
static size_t small_smem(int nf_max) { return ((size_t)P * nf_max + 2 * (size_t)P * kSmallCols) * sizeof(double); }

void solve_fwd_small(cudaStream_t s, const FrontDev &fd, const int *nodes, int n_nodes, int nf_max, const double *arena,
                     int k, double *X, int ldx) {
    if (n_nodes <= 0 || k <= 0) return;
    HSIM_SMEM_LIMIT_ONCE(k_solve_fwd_small<kSmallCols>, small_smem(kSmallNf));
    k_solve_fwd_small<kSmallCols><<<dim3((unsigned)n_nodes, cdiv(k, kSmallCols)), 256, small_smem(nf_max), s>>>(
        fd, nodes, arena, k, X, ldx, nf_max);
    HSIM_LAUNCHED();
}

void solve_bwd_small(cudaStream_t s, const FrontDev &fd, const int *nodes, int n_nodes, int nf_max, const double *arena,
                     int k, double *X, int ldx) {
    if (n_nodes <= 0 || k <= 0) return;
    HSIM_SMEM_LIMIT_ONCE(k_solve_bwd_small<kSmallCols>, small_smem(kSmallNf));
    k_solve_bwd_small<kSmallCols><<<dim3((unsigned)n_nodes, cdiv(k, kSmallCols)), 256, small_smem(nf_max), s>>>(
        fd, nodes, arena, k, X, ldx, nf_max);
    HSIM_LAUNCHED();
}

#define HSIM_FRONT_INSTANTIATE(T)                                                                                  \
    template void front_assemble<T>(cudaStream_t, int64_t, const int *, const int *, const int64_t *,            \
                                    const double *, const double *, const double *, double, T *);               \
    template void front_extend_add<T>(cudaStream_t, const FrontDev &, const int *, const int *, int, int, T *);  \
    template void front_panel<T>(cudaStream_t, const FrontDev &, const int *, int, int, int, T *, double, int *);  \
    template void front_update<T>(cudaStream_t, const FrontDev &, const int *, int, int, int, T *, int);         \
    template void front_maxdiag<T>(cudaStream_t, const FrontDev &, int, const T *, unsigned long long *);        \
    template void front_diag<T>(cudaStream_t, const FrontDev &, const int *, int, const T *, T *, int *);

HSIM_FRONT_INSTANTIATE(float)
HSIM_FRONT_INSTANTIATE(double)

}  // namespace k
}  // namespace hsim
