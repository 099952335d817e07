// Sparse kernels of the HSIM hot path: cotan/mass assembly (Sec. 3.1),
// CSR SpMM for S Psi, M Psi (Alg. 1) and the prolongation U Phi (Alg. 3),
// and the numeric Galerkin products U^T A U (Alg. 3), plus permutation and
// layout helpers.
//
// SpMM: one warp per sparse row (and 128-column block), lanes stride over the
// dense columns so every X row read is a contiguous segment; the row's nonzeros
// are broadcast from registers with warp shuffles.
#include <cuda_runtime.h>

#include <algorithm>

#include "common.h"
#include "fpconv.h"
#include "kernels.h"

namespace hsim {
namespace k {

namespace {

constexpr int kWarp = 32;

inline unsigned grid1d(int64_t work, int per_block) {
    int64_t g = (work + per_block - 1) / per_block;
    if (g < 1) g = 1;
    if (g > 2147483647LL) g = 2147483647LL;
    return (unsigned)g;
}

__global__ void k_triangle_geometry(int m, const int *__restrict__ F, const double *__restrict__ V,
                                    const double *__restrict__ L2, double *__restrict__ cot,
                                    double *__restrict__ area) {
    int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= m) return;
    double l[3];
    for (int k = 0; k < 3; ++k) {
        if (V) {
            const double *a = V + 3 * (size_t)F[3 * t + (k + 1) % 3];
            const double *b = V + 3 * (size_t)F[3 * t + (k + 2) % 3];
            double e0 = __dsub_rn(b[0], a[0]), e1 = __dsub_rn(b[1], a[1]), e2 = __dsub_rn(b[2], a[2]);
            l[k] = __dadd_rn(__dadd_rn(__dmul_rn(e0, e0), __dmul_rn(e1, e1)), __dmul_rn(e2, e2));
        } else {
            l[k] = L2[3 * (size_t)t + k];
        }
    }
    double s16 = 2.0 * (l[0] * l[1] + l[1] * l[2] + l[2] * l[0]) - (l[0] * l[0] + l[1] * l[1] + l[2] * l[2]);
    double A = 0.25 * sqrt(fmax(s16, 0.0));
    area[t] = A;
    for (int k = 0; k < 3; ++k)
        cot[3 * (size_t)t + k] = (l[(k + 1) % 3] + l[(k + 2) % 3] - l[k]) / (4.0 * A);
}

// ecot[2e], ecot[2e + 1]: corner indices 3 t + k of the (up to two)
// triangles t that hold edge e (-1 if none).  M: the lumped diagonal (n), or
// with `consistent` the consistent mass in S's pattern: A_t / 12 per
// triangle of an edge, A_t / 6 per triangle of the vertex on the diagonal.
__global__ void k_assemble_sm(int n, const int *__restrict__ ptr, const int *__restrict__ col,
                              const int *__restrict__ ecot, const double *__restrict__ cot,
                              const int *__restrict__ vt_ptr, const int *__restrict__ vt_idx,
                              const double *__restrict__ area, double *__restrict__ S,
                              double *__restrict__ M, bool consistent) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    double diag = 0.0;
    int de = -1;
    for (int e = ptr[i]; e < ptr[i + 1]; ++e) {
        if (col[e] == i) {
            de = e;
            continue;
        }
        double c = 0.0, me = 0.0;
        int a = ecot[2 * (size_t)e], b = ecot[2 * (size_t)e + 1];
        if (a >= 0) c += cot[a], me += area[a / 3] / 12.0;
        if (b >= 0) c += cot[b], me += area[b / 3] / 12.0;
        double v = -0.5 * c;
        S[e] = v;
        diag -= v;
        if (consistent) M[e] = me;
    }
    if (de >= 0) S[de] = diag;
    double mm = 0.0;
    for (int e = vt_ptr[i]; e < vt_ptr[i + 1]; ++e) mm += area[vt_idx[e]] / (consistent ? 6.0 : 3.0);
    if (!consistent) M[i] = mm;
    else if (de >= 0) M[de] = mm;
}

__global__ void k_row_sums(int n, const int *__restrict__ ptr, const double *__restrict__ val,
                           double *__restrict__ out) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    double s = 0.0;
    for (int e = ptr[i]; e < ptr[i + 1]; ++e) s += val[e];
    out[i] = s;
}

// Y = A X for narrow blocks, k <= 32 CH: one warp per row, lane l the columns l
// and l + 32, the row's entries broadcast from registers four at a time so that
// the gathers of four X rows are in flight together.
template <int CH>
__global__ void __launch_bounds__(128) k_spmm_narrow(int n_rows, const int *__restrict__ ptr, const int *__restrict__ col,
                                                     const double *__restrict__ val, int k, const double *__restrict__ X,
                                                     int ldx, double *__restrict__ Y, int ldy) {
    const int lane = threadIdx.x & 31;
    const int64_t row = (int64_t)blockIdx.x * 4 + (threadIdx.x >> 5);
    if (row >= n_rows) return;
    const int beg = ptr[row], end = ptr[row + 1];
    double acc[CH];
#pragma unroll
    for (int u = 0; u < CH; ++u) acc[u] = 0.0;
    for (int e0 = beg; e0 < end; e0 += 32) {
        int my_c = 0;
        double my_v = 0.0;
        if (e0 + lane < end) {
            my_c = col[e0 + lane];
            my_v = val[e0 + lane];
        }
        const int cnt = min(32, end - e0);
        for (int t0 = 0; t0 < cnt; t0 += 4) {
            double x[4][CH];
#pragma unroll
            for (int t = 0; t < 4; ++t) {
                const double *xr = X + (size_t)__shfl_sync(0xffffffffu, my_c, (t0 + t) & 31) * ldx + lane;
#pragma unroll
                for (int u = 0; u < CH; ++u) x[t][u] = t0 + t < cnt && 32 * u + lane < k ? xr[32 * u] : 0.0;
            }
#pragma unroll
            for (int t = 0; t < 4; ++t) {
                const double v = __shfl_sync(0xffffffffu, my_v, (t0 + t) & 31);
                if (t0 + t >= cnt) break;
#pragma unroll
                for (int u = 0; u < CH; ++u) acc[u] = fma(v, x[t][u], acc[u]);
            }
        }
    }
    double *yr = Y + (size_t)row * ldy + lane;
#pragma unroll
    for (int u = 0; u < CH; ++u)
        if (32 * u + lane < k) yr[32 * u] = acc[u];
}

constexpr int kSpmmRows = 16;  // rows (warps) per CTA of the column-block SpMM

// Y = A X for k > 64: a CTA takes 16 consecutive rows of one 128-column block,
// the column block the slow index: the CTA's gathered 1 KB row segments stay in
// L1, and concurrently running CTAs share the same column block in L2.  Bound by
// the FP64 pipe, 1.86 of nominally 2 lanes per clock and SM at 10^6 rows x 750 (9.0
// ms), where an instruction costs a warp the same time however many lanes it serves.
// Two layouts of a block on the lanes:
// k_spmm4: four consecutive columns per lane, read as pairs (every block at
//   least 97 columns wide: nothing to skip; 0.5 to 1 % faster than the other);
// k_spmm_groups: columns l, l + 32, l + 64, l + 96, groups of 32 beyond k skipped
//   (75 columns: three of four groups).
template <int NG>
__device__ __forceinline__ void spmm_block(const int *__restrict__ col, const double *__restrict__ val, int beg, int end,
                                           const double *__restrict__ X, int ldx, bool last, double *__restrict__ y) {
    const int lane = threadIdx.x & 31;
    double acc[NG];
#pragma unroll
    for (int v = 0; v < NG; ++v) acc[v] = 0.0;
    for (int e0 = beg; e0 < end; e0 += 32) {
        int my_c = 0;
        double my_v = 0.0;
        if (e0 + lane < end) {
            my_c = col[e0 + lane];
            my_v = val[e0 + lane];
        }
        const int cnt = min(32, end - e0);
        auto load = [&](int t, double (&x)[NG]) {
            const double *xr = X + (size_t)__shfl_sync(0xffffffffu, my_c, t) * ldx;
#pragma unroll
            for (int v = 0; v < NG; ++v) x[v] = v < NG - 1 || last ? xr[32 * v] : 0.0;
        };
        int t = 0;
        for (; t + 1 < cnt; t += 2) {
            double xa[NG], xb[NG];
            load(t, xa);
            load(t + 1, xb);
            const double sa = __shfl_sync(0xffffffffu, my_v, t), sb = __shfl_sync(0xffffffffu, my_v, t + 1);
#pragma unroll
            for (int v = 0; v < NG; ++v) acc[v] = fma(sa, xa[v], acc[v]);
#pragma unroll
            for (int v = 0; v < NG; ++v) acc[v] = fma(sb, xb[v], acc[v]);
        }
        if (t < cnt) {
            double xa[NG];
            load(t, xa);
            const double sa = __shfl_sync(0xffffffffu, my_v, t);
#pragma unroll
            for (int v = 0; v < NG; ++v) acc[v] = fma(sa, xa[v], acc[v]);
        }
    }
#pragma unroll
    for (int v = 0; v < NG; ++v)
        if (v < NG - 1 || last) y[32 * v] = acc[v];
}

__global__ void __launch_bounds__(kSpmmRows * 32) k_spmm_groups(int n_rows, const int *__restrict__ ptr,
                                                                const int *__restrict__ col,
                                                                const double *__restrict__ val, int k,
                                                                const double *__restrict__ X, int ldx,
                                                                double *__restrict__ Y, int ldy) {
    const int nrg = (n_rows + kSpmmRows - 1) / kSpmmRows;
    const int cb = blockIdx.x / nrg, row = (blockIdx.x - cb * nrg) * kSpmmRows + (threadIdx.x >> 5);
    if (row >= n_rows) return;
    const int c = cb * 128 + (threadIdx.x & 31), ng = min(4, (k - cb * 128 + 31) / 32);
    const bool last = c + 32 * (ng - 1) < k;  // this lane's column of the last group
    const int beg = ptr[row], end = ptr[row + 1];
    double *y = Y + (size_t)row * ldy + c;
    if (ng == 4) spmm_block<4>(col, val, beg, end, X + c, ldx, last, y);
    else if (ng == 3) spmm_block<3>(col, val, beg, end, X + c, ldx, last, y);
    else if (ng == 2) spmm_block<2>(col, val, beg, end, X + c, ldx, last, y);
    else spmm_block<1>(col, val, beg, end, X + c, ldx, last, y);
}

__device__ __forceinline__ void load_d4(double (&x)[4], const double *__restrict__ X, int r, int c, int k, int ldx,
                                        bool vec) {
    const double *p = X + (size_t)r * ldx + c;
    if (vec && c + 4 <= k) {
        const double2 a = reinterpret_cast<const double2 *>(p)[0], b = reinterpret_cast<const double2 *>(p)[1];
        x[0] = a.x, x[1] = a.y, x[2] = b.x, x[3] = b.y;
    } else {
#pragma unroll
        for (int v = 0; v < 4; ++v) x[v] = c + v < k ? p[v] : 0.0;
    }
}

__global__ void __launch_bounds__(kSpmmRows * 32) k_spmm4(int n_rows, const int *__restrict__ ptr,
                                                          const int *__restrict__ col, const double *__restrict__ val,
                                                          int k, const double *__restrict__ X, int ldx,
                                                          double *__restrict__ Y, int ldy, bool vec) {
    const int lane = threadIdx.x & 31;
    const int nrg = (n_rows + kSpmmRows - 1) / kSpmmRows;
    const int cb = blockIdx.x / nrg, row = (blockIdx.x - cb * nrg) * kSpmmRows + (threadIdx.x >> 5);
    const int c = cb * 128 + lane * 4;
    if (row >= n_rows) return;
    double acc[4] = {0.0, 0.0, 0.0, 0.0};
    const int beg = ptr[row], end = ptr[row + 1];
    for (int e0 = beg; e0 < end; e0 += 32) {
        int my_c = 0;
        double my_v = 0.0;
        if (e0 + lane < end) {
            my_c = col[e0 + lane];
            my_v = val[e0 + lane];
        }
        const int cnt = min(32, end - e0);
        int t = 0;
        for (; t + 1 < cnt; t += 2) {
            const int ca = __shfl_sync(0xffffffffu, my_c, t), cb2 = __shfl_sync(0xffffffffu, my_c, t + 1);
            const double sa = __shfl_sync(0xffffffffu, my_v, t), sb = __shfl_sync(0xffffffffu, my_v, t + 1);
            double xa[4], xb[4];
            load_d4(xa, X, ca, c, k, ldx, vec);
            load_d4(xb, X, cb2, c, k, ldx, vec);
#pragma unroll
            for (int v = 0; v < 4; ++v) acc[v] = fma(sa, xa[v], acc[v]);
#pragma unroll
            for (int v = 0; v < 4; ++v) acc[v] = fma(sb, xb[v], acc[v]);
        }
        if (t < cnt) {
            const int ca = __shfl_sync(0xffffffffu, my_c, t);
            const double sa = __shfl_sync(0xffffffffu, my_v, t);
            double xa[4];
            load_d4(xa, X, ca, c, k, ldx, vec);
#pragma unroll
            for (int v = 0; v < 4; ++v) acc[v] = fma(sa, xa[v], acc[v]);
        }
    }
    double *yr = Y + (size_t)row * ldy;
#pragma unroll
    for (int v = 0; v < 4; ++v)
        if (c + v < k) yr[c + v] = acc[v];
}

// R[r, :] = B[r, :] - sum_e (S_e - mu M_e) X[col_e, :]  (M in S's pattern, or a
// diagonal Md); the residual of the shifted system for iterative refinement
template <int kChunk>
__global__ void k_shifted_residual(int n_rows, const int *__restrict__ ptr, const int *__restrict__ col,
                                   const double *__restrict__ S, const double *__restrict__ M,
                                   const double *__restrict__ Md, double mu, int k, const double *__restrict__ X,
                                   int ldx, const double *__restrict__ B, int ldb, double *__restrict__ R, int ldr) {
    const int lane = threadIdx.x & (kWarp - 1);
    const int warps = blockDim.x / kWarp;
    int64_t row = (int64_t)blockIdx.x * warps + threadIdx.x / kWarp;
    if (row >= n_rows) return;
    const int beg = ptr[row], end = ptr[row + 1];
    for (int c0 = 0; c0 < k; c0 += kChunk * kWarp) {
        double acc[kChunk];
#pragma unroll
        for (int u = 0; u < kChunk; ++u) acc[u] = 0.0;
        for (int e0 = beg; e0 < end; e0 += kWarp) {
            int my_c = 0;
            double my_v = 0.0;
            if (e0 + lane < end) {
                my_c = col[e0 + lane];
                my_v = S[e0 + lane];
                if (M) my_v -= mu * M[e0 + lane];
                else if (my_c == row) my_v -= mu * Md[row];
            }
            const int cnt = min(kWarp, end - e0);
            for (int t = 0; t < cnt; ++t) {
                int c = __shfl_sync(0xffffffffu, my_c, t);
                double v = __shfl_sync(0xffffffffu, my_v, t);
                const double *xr = X + (size_t)c * ldx;
#pragma unroll
                for (int u = 0; u < kChunk; ++u) {
                    int j = c0 + u * kWarp + lane;
                    if (j < k) acc[u] += v * xr[j];
                }
            }
        }
#pragma unroll
        for (int u = 0; u < kChunk; ++u) {
            int j = c0 + u * kWarp + lane;
            if (j < k) R[(size_t)row * ldr + j] = B[(size_t)row * ldb + j] - acc[u];
        }
    }
}

__global__ void k_axpy_matrix(int n, int k, const double *__restrict__ X, int ldx, double *__restrict__ Y, int ldy) {
    HSIM_FOR_RC(i, n, j, k) Y[(size_t)i * ldy + j] += X[(size_t)i * ldx + j];
}

__global__ void k_diag_scale(int n, int k, const double *__restrict__ d, const double *__restrict__ X, int ldx,
                             double *__restrict__ Y, int ldy) {
    HSIM_ROWS_OF_COLUMN(i, n, j, k) Y[(size_t)i * ldy + j] = d[i] * X[(size_t)i * ldx + j];
}

__device__ __forceinline__ int find_col(const int *__restrict__ c, int lo, int hi, int key) {
    // position of key in the sorted range c[lo, hi), or -1
    const int end = hi;
    while (lo < hi) {
        int mid = (lo + hi) >> 1;
        if (c[mid] < key) lo = mid + 1;
        else hi = mid;
    }
    return (lo < end && c[lo] == key) ? lo : -1;
}

// T[i, j] = sum_k A[i,k] U[k,j] for every (i, j) of T's pattern; one warp per
// row, one lane per output entry.
__global__ void k_galerkin_au(int n, const int *__restrict__ a_ptr, const int *__restrict__ a_col,
                              const double *__restrict__ a_val, const int *__restrict__ u_ptr,
                              const int *__restrict__ u_col, const double *__restrict__ u_val,
                              const int *__restrict__ t_ptr, const int *__restrict__ t_col,
                              double *__restrict__ t_val) {
    const int lane = threadIdx.x & (kWarp - 1);
    int64_t i = (int64_t)blockIdx.x * (blockDim.x / kWarp) + threadIdx.x / kWarp;
    if (i >= n) return;
    for (int e = t_ptr[i] + lane; e < t_ptr[i + 1]; e += kWarp) {
        int j = t_col[e];
        double acc = 0.0;
        for (int f = a_ptr[i]; f < a_ptr[i + 1]; ++f) {
            int kk = a_col[f];
            int pos = find_col(u_col, u_ptr[kk], u_ptr[kk + 1], j);
            if (pos >= 0) acc += a_val[f] * u_val[pos];
        }
        t_val[e] = acc;
    }
}

__global__ void k_galerkin_utt(int nc, const int *__restrict__ ut_ptr, const int *__restrict__ ut_col,
                               const double *__restrict__ ut_val, const int *__restrict__ t_ptr,
                               const int *__restrict__ t_col, const double *__restrict__ t_val,
                               const int *__restrict__ c_ptr, const int *__restrict__ c_col,
                               double *__restrict__ c_val) {
    const int lane = threadIdx.x & (kWarp - 1);
    int64_t a = (int64_t)blockIdx.x * (blockDim.x / kWarp) + threadIdx.x / kWarp;
    if (a >= nc) return;
    for (int e = c_ptr[a] + lane; e < c_ptr[a + 1]; e += kWarp) {
        int b = c_col[e];
        double acc = 0.0;
        for (int f = ut_ptr[a]; f < ut_ptr[a + 1]; ++f) {
            int i = ut_col[f];
            int pos = find_col(t_col, t_ptr[i], t_ptr[i + 1], b);
            if (pos >= 0) acc += ut_val[f] * t_val[pos];
        }
        c_val[e] = acc;
    }
}

__global__ void k_gather_values(int64_t n, const int64_t *__restrict__ map, const double *__restrict__ in,
                                double *__restrict__ out) {
    int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e < n) out[e] = in[map[e]];
}
__global__ void k_gather_values_i(int64_t n, const int *__restrict__ map, const double *__restrict__ in,
                                  double *__restrict__ out) {
    int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e < n) out[e] = in[map[e]];
}

__global__ void k_gather_rows(int n, int k, const int *__restrict__ perm, const double *__restrict__ X, int ldx,
                              double *__restrict__ Y, int ldy) {
    HSIM_FOR_RC(i, n, j, k) Y[(size_t)i * ldy + j] = X[(size_t)perm[i] * ldx + j];
}

__global__ void k_copy_matrix(int rows, int cols, const double *__restrict__ X, int ldx, double *__restrict__ Y,
                              int ldy) {
    HSIM_ROWS_OF_COLUMN(i, rows, j, cols) Y[(size_t)i * ldy + j] = X[(size_t)i * ldx + j];
}

__global__ void k_densify(int n, const int *__restrict__ ptr, const int *__restrict__ col,
                          const double *__restrict__ val, double *__restrict__ D) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    for (int e = ptr[i]; e < ptr[i + 1]; ++e) D[(size_t)i * n + col[e]] = val[e];
}
__global__ void k_densify_diag(int n, const double *__restrict__ d, double *__restrict__ D) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) D[(size_t)i * n + i] = d[i];
}

// per column j: index of the entry of largest magnitude (lowest row on ties),
// reduced over rows by one block per column
__global__ void k_col_sign(int n, const double *__restrict__ Phi, int ldp, double *__restrict__ sign) {
    int j = blockIdx.x;
    double best = -1.0, bv = 0.0;
    int bi = 0x7fffffff;
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        double v = Phi[(size_t)i * ldp + j];
        double a = fabs(v);
        if (a > best || (a == best && i < bi)) { best = a; bi = i; bv = v; }
    }
    __shared__ double sb[256], sv[256];
    __shared__ int si[256];
    sb[threadIdx.x] = best;
    sv[threadIdx.x] = bv;
    si[threadIdx.x] = bi;
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
        if (threadIdx.x < w) {
            int o = threadIdx.x + w;
            if (sb[o] > sb[threadIdx.x] || (sb[o] == sb[threadIdx.x] && si[o] < si[threadIdx.x])) {
                sb[threadIdx.x] = sb[o];
                sv[threadIdx.x] = sv[o];
                si[threadIdx.x] = si[o];
            }
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) sign[j] = sv[0] < 0.0 ? -1.0 : 1.0;
}

__global__ void k_output_evecs(int n, int p, const int *__restrict__ iperm, const double *__restrict__ Phi, int ldp,
                               const double *__restrict__ sign, double *__restrict__ out) {
    int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (int64_t)n * p) return;
    int j = (int)(idx / n), i = (int)(idx % n);
    int r = iperm ? iperm[i] : i;
    out[idx] = sign[j] * Phi[(size_t)r * ldp + j];
}

__global__ void k_reciprocal(int n, const double *__restrict__ x, double *__restrict__ y) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) y[i] = 1.0 / x[i];
}

template <typename Tin, typename Tout>
__global__ void k_convert_matrix(int rows, int cols, const Tin *__restrict__ X, int ldx, Tout *__restrict__ Y, int ldy) {
    int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (int64_t)rows * cols) return;
    int i = (int)(idx / cols), j = (int)(idx % cols);
    Y[(size_t)i * ldy + j] = (Tout)X[(size_t)i * ldx + j];
}


// rho_j = num[j] / den[j] (den NULL: rho_j = num[j]), once per column
__global__ void k_rho(int cols, const double *__restrict__ num, const double *__restrict__ den,
                      double *__restrict__ rho) {
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j < cols) rho[j] = den ? num[j] / den[j] : num[j];
}

// R (FP32) = SP - rho_j MP: the difference in FP64 (it cancels), then
// truncated to FP32
__global__ void k_residual_f32(int rows, int cols, const double *__restrict__ SP, int lds,
                               const double *__restrict__ MP, int ldm, const double *__restrict__ rho,
                               float *__restrict__ R, int ldr) {
    const double rj = rho[min((int)(blockIdx.x * blockDim.x + threadIdx.x), cols - 1)];
    HSIM_ROWS_OF_COLUMN(i, rows, j, cols) R[(size_t)i * ldr + j] =
        d2f_trunc(fma(-rj, MP[(size_t)i * ldm + j], SP[(size_t)i * lds + j]));
}

// R (FP32) = SP - rho_j m_i X with M = diag(m): M X is not formed
__global__ void k_residual_f32_diag(int rows, int cols, const double *__restrict__ SP, int lds,
                                    const double *__restrict__ X, int ldx, const double *__restrict__ m,
                                    const double *__restrict__ rho, float *__restrict__ R, int ldr) {
    const double rj = rho[min((int)(blockIdx.x * blockDim.x + threadIdx.x), cols - 1)];
    HSIM_ROWS_OF_COLUMN(i, rows, j, cols) R[(size_t)i * ldr + j] =
        d2f_trunc(fma(-rj * m[i], X[(size_t)i * ldx + j], SP[(size_t)i * lds + j]));
}

// Y (FP64) = X - Z (FP32)
__global__ void k_sub_f2d(int rows, int cols, const double *__restrict__ X, int ldx, const float *__restrict__ Z,
                          int ldz, double *__restrict__ Y, int ldy) {
    HSIM_ROWS_OF_COLUMN(i, rows, j, cols) Y[(size_t)i * ldy + j] = X[(size_t)i * ldx + j] - f2d_bits(Z[(size_t)i * ldz + j]);
}

template <typename T>
__global__ void k_copy_matrix_t(int rows, int cols, const T *__restrict__ X, int ldx, T *__restrict__ Y, int ldy) {
    int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (int64_t)rows * cols) return;
    int i = (int)(idx / cols), j = (int)(idx % cols);
    Y[(size_t)i * ldy + j] = X[(size_t)i * ldx + j];
}

__global__ void k_diag_scale_f(int n, int k, const float *__restrict__ d, const float *__restrict__ X, int ldx,
                               float *__restrict__ Y, int ldy) {
    int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (int64_t)n * k) return;
    int i = (int)(idx / k), j = (int)(idx % k);
    Y[(size_t)i * ldy + j] = d[i] * X[(size_t)i * ldx + j];
}

__global__ void k_f2d(int64_t n, const float *__restrict__ x, double *__restrict__ y) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) y[i] = (double)x[i];
}
__global__ void k_d2f(int64_t n, const double *__restrict__ x, float *__restrict__ y) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) y[i] = (float)x[i];
}

}  // namespace

void triangle_geometry(cudaStream_t s, int m, const int *F, const double *V, const double *L2, double *cot,
                       double *area) {
    k_triangle_geometry<<<grid1d(m, 256), 256, 0, s>>>(m, F, V, L2, cot, area);
    HSIM_LAUNCHED();
}

void row_sums(cudaStream_t s, int n, const int *ptr, const double *val, double *out) {
    if (n <= 0) return;
    k_row_sums<<<grid1d(n, 256), 256, 0, s>>>(n, ptr, val, out);
    HSIM_LAUNCHED();
}

void assemble_sm(cudaStream_t s, int n, const int *ptr, const int *col, const int *ecot, const double *cot,
                 const int *vt_ptr, const int *vt_idx, const double *area, double *S_val, double *M_diag,
                 bool consistent) {
    k_assemble_sm<<<grid1d(n, 256), 256, 0, s>>>(n, ptr, col, ecot, cot, vt_ptr, vt_idx, area, S_val, M_diag,
                                                 consistent);
    HSIM_LAUNCHED();
}

void spmm(cudaStream_t s, int n_rows, const int *ptr, const int *col, const double *val, int k, const double *X,
          int ldx, double *Y, int ldy) {
    if (n_rows <= 0 || k <= 0) return;
    if (k > 64) {
        // wide blocks: column-block mapping (L1 reuse of the gathered rows)
        const unsigned blocks = (unsigned)(((n_rows + kSpmmRows - 1) / kSpmmRows) * ((k + 127) / 128));
        const bool vec = (reinterpret_cast<uintptr_t>(X) % 16 == 0) && (ldx % 2 == 0);
        if (k % 128 == 0 || k % 128 > 96)
            k_spmm4<<<blocks, kSpmmRows * 32, 0, s>>>(n_rows, ptr, col, val, k, X, ldx, Y, ldy, vec);
        else
            k_spmm_groups<<<blocks, kSpmmRows * 32, 0, s>>>(n_rows, ptr, col, val, k, X, ldx, Y, ldy);
    } else if (k > 32) {
        k_spmm_narrow<2><<<grid1d(n_rows, 4), 128, 0, s>>>(n_rows, ptr, col, val, k, X, ldx, Y, ldy);
    } else {
        k_spmm_narrow<1><<<grid1d(n_rows, 4), 128, 0, s>>>(n_rows, ptr, col, val, k, X, ldx, Y, ldy);
    }
    HSIM_LAUNCHED();
}



void shifted_residual(cudaStream_t s, int n_rows, const int *ptr, const int *col, const double *S, const double *M,
                      const double *Md, double mu, int k, const double *X, int ldx, const double *B, int ldb,
                      double *R, int ldr) {
    if (n_rows <= 0 || k <= 0) return;
    const int warps = 8;
    unsigned g = grid1d(n_rows, warps);
    if (k <= 32 * 8)
        k_shifted_residual<8><<<g, warps * 32, 0, s>>>(n_rows, ptr, col, S, M, Md, mu, k, X, ldx, B, ldb, R, ldr);
    else
        k_shifted_residual<24><<<g, warps * 32, 0, s>>>(n_rows, ptr, col, S, M, Md, mu, k, X, ldx, B, ldb, R, ldr);
    HSIM_LAUNCHED();
}

void axpy_matrix(cudaStream_t s, int n, int k, const double *X, int ldx, double *Y, int ldy) {
    if (n <= 0 || k <= 0) return;
    k_axpy_matrix<<<grid_rc(n, k), 256, 0, s>>>(n, k, X, ldx, Y, ldy);
    HSIM_LAUNCHED();
}

void diag_scale(cudaStream_t s, int n, int k, const double *d, const double *X, int ldx, double *Y, int ldy) {
    if (n <= 0 || k <= 0) return;
    k_diag_scale<<<grid_rc(n, k), 256, 0, s>>>(n, k, d, X, ldx, Y, ldy);
    HSIM_LAUNCHED();
}

void galerkin_au(cudaStream_t s, int n, const int *a_ptr, const int *a_col, const double *a_val, const int *u_ptr,
                 const int *u_col, const double *u_val, const int *t_ptr, const int *t_col, double *t_val) {
    k_galerkin_au<<<grid1d(n, 8), 256, 0, s>>>(n, a_ptr, a_col, a_val, u_ptr, u_col, u_val, t_ptr, t_col, t_val);
    HSIM_LAUNCHED();
}

void galerkin_utt(cudaStream_t s, int nc, const int *ut_ptr, const int *ut_col, const double *ut_val,
                  const int *t_ptr, const int *t_col, const double *t_val, const int *c_ptr, const int *c_col,
                  double *c_val) {
    k_galerkin_utt<<<grid1d(nc, 8), 256, 0, s>>>(nc, ut_ptr, ut_col, ut_val, t_ptr, t_col, t_val, c_ptr, c_col,
                                                 c_val);
    HSIM_LAUNCHED();
}

void gather_values(cudaStream_t s, int64_t n, const int64_t *map, const double *in, double *out) {
    if (n <= 0) return;
    k_gather_values<<<grid1d(n, 256), 256, 0, s>>>(n, map, in, out);
    HSIM_LAUNCHED();
}
void gather_values_i(cudaStream_t s, int64_t n, const int *map, const double *in, double *out) {
    if (n <= 0) return;
    k_gather_values_i<<<grid1d(n, 256), 256, 0, s>>>(n, map, in, out);
    HSIM_LAUNCHED();
}

void gather_rows(cudaStream_t s, int n, int k, const int *perm, const double *X, int ldx, double *Y, int ldy) {
    if (n <= 0 || k <= 0) return;
    k_gather_rows<<<grid_rc(n, k), 256, 0, s>>>(n, k, perm, X, ldx, Y, ldy);
    HSIM_LAUNCHED();
}

void copy_matrix(cudaStream_t s, int rows, int cols, const double *X, int ldx, double *Y, int ldy) {
    if (rows <= 0 || cols <= 0) return;
    k_copy_matrix<<<grid_rc(rows, cols), 256, 0, s>>>(rows, cols, X, ldx, Y, ldy);
    HSIM_LAUNCHED();
}

void densify(cudaStream_t s, int n, const int *ptr, const int *col, const double *val, double *D) {
    HSIM_CUDA(cudaMemsetAsync(D, 0, (size_t)n * n * sizeof(double), s));
    k_densify<<<grid1d(n, 128), 128, 0, s>>>(n, ptr, col, val, D);
    HSIM_LAUNCHED();
}
void densify_diag(cudaStream_t s, int n, const double *d, double *D) {
    HSIM_CUDA(cudaMemsetAsync(D, 0, (size_t)n * n * sizeof(double), s));
    k_densify_diag<<<grid1d(n, 128), 128, 0, s>>>(n, d, D);
    HSIM_LAUNCHED();
}

void output_evecs(cudaStream_t s, int n, int p, const int *iperm, const double *Phi, int ldp, double *out,
                  double *scratch_p) {
    if (n <= 0 || p <= 0) return;
    // the sign is decided on the internal-order rows; the entry of largest
    // magnitude is the same entry whichever order the rows are in, up to ties
    k_col_sign<<<p, 256, 0, s>>>(n, Phi, ldp, scratch_p);
    HSIM_LAUNCHED();
    k_output_evecs<<<grid1d((int64_t)n * p, 256), 256, 0, s>>>(n, p, iperm, Phi, ldp, scratch_p, out);
    HSIM_LAUNCHED();
}

void convert_matrix(cudaStream_t s, int rows, int cols, const double *X, int ldx, float *Y, int ldy) {
    if (rows <= 0 || cols <= 0) return;
    k_convert_matrix<double, float><<<grid1d((int64_t)rows * cols, 256), 256, 0, s>>>(rows, cols, X, ldx, Y, ldy);
    HSIM_LAUNCHED();
}
void convert_matrix(cudaStream_t s, int rows, int cols, const float *X, int ldx, double *Y, int ldy) {
    if (rows <= 0 || cols <= 0) return;
    k_convert_matrix<float, double><<<grid1d((int64_t)rows * cols, 256), 256, 0, s>>>(rows, cols, X, ldx, Y, ldy);
    HSIM_LAUNCHED();
}
void residual_f32(cudaStream_t s, int rows, int cols, const double *SP, int lds, const double *MP, int ldm,
                  const double *num, const double *den, double *rho, float *R, int ldr) {
    if (rows <= 0 || cols <= 0) return;
    k_rho<<<(cols + 255) / 256, 256, 0, s>>>(cols, num, den, rho);
    HSIM_LAUNCHED();
    k_residual_f32<<<grid_rc(rows, cols), 256, 0, s>>>(rows, cols, SP, lds, MP, ldm, rho, R, ldr);
    HSIM_LAUNCHED();
}
void residual_f32_diag(cudaStream_t s, int rows, int cols, const double *SP, int lds, const double *X, int ldx,
                       const double *m, const double *num, const double *den, double *rho, float *R, int ldr) {
    if (rows <= 0 || cols <= 0) return;
    k_rho<<<(cols + 255) / 256, 256, 0, s>>>(cols, num, den, rho);
    HSIM_LAUNCHED();
    k_residual_f32_diag<<<grid_rc(rows, cols), 256, 0, s>>>(rows, cols, SP, lds, X, ldx, m, rho, R, ldr);
    HSIM_LAUNCHED();
}
void sub_f2d(cudaStream_t s, int rows, int cols, const double *X, int ldx, const float *Z, int ldz, double *Y,
             int ldy) {
    if (rows <= 0 || cols <= 0) return;
    k_sub_f2d<<<grid_rc(rows, cols), 256, 0, s>>>(rows, cols, X, ldx, Z, ldz, Y, ldy);
    HSIM_LAUNCHED();
}
void copy_matrix(cudaStream_t s, int rows, int cols, const float *X, int ldx, float *Y, int ldy) {
    if (rows <= 0 || cols <= 0) return;
    k_copy_matrix_t<float><<<grid1d((int64_t)rows * cols, 256), 256, 0, s>>>(rows, cols, X, ldx, Y, ldy);
    HSIM_LAUNCHED();
}
void diag_scale(cudaStream_t s, int n, int k, const float *d, const float *X, int ldx, float *Y, int ldy) {
    if (n <= 0 || k <= 0) return;
    k_diag_scale_f<<<grid1d((int64_t)n * k, 256), 256, 0, s>>>(n, k, d, X, ldx, Y, ldy);
    HSIM_LAUNCHED();
}

void reciprocal(cudaStream_t s, int n, const double *x, double *y) {
    if (n <= 0) return;
    k_reciprocal<<<grid1d(n, 256), 256, 0, s>>>(n, x, y);
    HSIM_LAUNCHED();
}

void convert_f2d(cudaStream_t s, int64_t n, const float *x, double *y) {
    if (n <= 0) return;
    k_f2d<<<grid1d(n, 256), 256, 0, s>>>(n, x, y);
    HSIM_LAUNCHED();
}
void convert_d2f(cudaStream_t s, int64_t n, const double *x, float *y) {
    if (n <= 0) return;
    k_d2f<<<grid1d(n, 256), 256, 0, s>>>(n, x, y);
    HSIM_LAUNCHED();
}

}  // namespace k
}  // namespace hsim
