// Shape gradient of a loss of the eigenvalues (first-order perturbation of
// S Phi = lambda M Phi for M-normalised eigenvectors, applied to the cotan
// stiffness and lumped mass of Sec. 3.1):
//
//     dL/dx_v = sum_i w_i phi_i^T (dS/dx_v - lambda_i dM/dx_v) phi_i,
//     w_i = dL/dlambda_i.
//
// Per triangle with corners x_0, x_1, x_2 the quadratic forms are
//     phi^T S phi |_t = 1/2 sum_k cot_k (phi_{k+1} - phi_{k+2})^2,
//     phi^T M phi |_t = A_t / 3 sum_k phi_k^2,
// so one pass over the eigenpairs reduces every triangle to four numbers,
//     D_k = sum_i w_i (phi_i(k+1) - phi_i(k+2))^2,  P = sum of the corners' P_v,
//     P_v = sum_i w_i lambda_i phi_i(v)^2 (once per vertex, k_vertex_energy),
// and its part of the loss is E = sum_k t_k D_k / (2 s) - P s / 6 with the edges
// e_0 = x_2 - x_1, e_1 = x_0 - x_2, e_2 = x_1 - x_0, t_k = -e_{k+1}.e_{k+2} (the
// corner's u.w), s = |u x w| = 2 A, cot_k = t_k / s.  In the squared lengths l_k
// = e_k.e_k, t_k = (l_{k+1} + l_{k+2} - l_k) / 2, and with the unit normal N = e_1 x
// e_2 / s the derivative of s by corner k is N x e_k, so
//     dE/dx_k = c_{k+1} e_{k+1} - c_{k+2} e_{k+2} + E_s N x e_k,
//     c_k = (D_{k+1} + D_{k+2} - D_k) / (2 s),  E_s = -sum_k t_k D_k / (2 s^2) - P / 6
// (and dE/dx_2 = -dE/dx_0 - dE/dx_1).  N x e_k is taken as a cross product: the same
// vector as the difference (t_{k+1} e_{k+1} - t_{k+2} e_{k+2}) / s has four times the
// rounding error in a flat obtuse triangle, where the two edges nearly cancel.
// One thread per triangle; the nine partial derivatives go to the vertices
// with FP64 atomics (the order of the additions, hence the last bits, vary
// from run to run).
//
// What bounds it: FP64 instructions (1.7 to 1.9 lanes per clock and SM), nine per
// triangle and eigenpair, two per vertex and eigenpair and about 100 per
// triangle: 80,000 triangles x 50 pairs take 93 + 12 us, where fourteen (P per triangle)
// and the derivatives of the three cotangents one by one took 206 us.  CTAs of 64
// threads spread 1,250 over 152 SMs evenly; of 256 threads 313 left a third of
// them a CTA behind.

#include "common.h"
#include "kernels.h"

namespace hsim {
namespace k {

namespace {

struct v3 {
    double x, y, z;
};
__device__ __forceinline__ v3 sub(v3 a, v3 b) { return {a.x - b.x, a.y - b.y, a.z - b.z}; }
__device__ __forceinline__ v3 add(v3 a, v3 b) { return {a.x + b.x, a.y + b.y, a.z + b.z}; }
__device__ __forceinline__ v3 mul(double s, v3 a) { return {s * a.x, s * a.y, s * a.z}; }
__device__ __forceinline__ double dot(v3 a, v3 b) { return a.x * b.x + a.y * b.y + a.z * b.z; }
__device__ __forceinline__ v3 cross(v3 a, v3 b) {
    return {a.y * b.z - a.z * b.y, a.z * b.x - a.x * b.z, a.x * b.y - a.y * b.x};
}
// x == 0 on the bits (the FP64 comparison takes its place in the FP64 pipe)
__device__ __forceinline__ bool is_zero(double x) { return (__double_as_longlong(x) << 1) == 0; }
__device__ __forceinline__ v3 load(const double *V, int v) {
    return {V[3 * (size_t)v], V[3 * (size_t)v + 1], V[3 * (size_t)v + 2]};
}
__device__ __forceinline__ void atomic_add3(double *g, int v, v3 a) {
    atomicAdd(g + 3 * (size_t)v, a.x);
    atomicAdd(g + 3 * (size_t)v + 1, a.y);
    atomicAdd(g + 3 * (size_t)v + 2, a.z);
}

// Pv[v] = sum_i w_i lambda_i phi_i(v)^2
__global__ void __launch_bounds__(64) k_vertex_energy(int n, int p, const double *__restrict__ evals,
                                                      const double *__restrict__ evecs, int ld,
                                                      const double *__restrict__ dl, double *__restrict__ Pv) {
    __shared__ double wl[64];
    const int v = blockIdx.x * blockDim.x + threadIdx.x;
    const double *f = evecs + min(v, n - 1);
    double P = 0.0;
    for (int i0 = 0; i0 < p; i0 += 64) {
        const int cnt = min(64, p - i0);
        __syncthreads();
        if ((int)threadIdx.x < cnt) wl[threadIdx.x] = __ldg(dl + i0 + threadIdx.x) * __ldg(evals + i0 + threadIdx.x);
        __syncthreads();
#pragma unroll 8
        for (int i = 0; i < cnt; ++i) {
            const double x = __ldg(f + (size_t)(i0 + i) * ld);
            if (!is_zero(__ldg(dl + i0 + i))) P = fma(wl[i] * x, x, P);
        }
    }
    if (v < n) Pv[v] = P;
}

__global__ void __launch_bounds__(64) k_eig_grad(int m, int p, const double *__restrict__ V, const int *__restrict__ F,
                                                 const double *__restrict__ evecs, int ld,
                                                 const double *__restrict__ dl, const double *__restrict__ Pv,
                                                 double *__restrict__ g) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= m) return;
    const int c[3] = {F[3 * (size_t)t], F[3 * (size_t)t + 1], F[3 * (size_t)t + 2]};
    double D0 = 0.0, D1 = 0.0, D2 = 0.0;
    const double *q0 = evecs + c[0], *q1 = evecs + c[1], *q2 = evecs + c[2];
#pragma unroll 4
    for (int i = 0; i < p; ++i) {
        const double w = __ldg(dl + i);
        const double f0 = __ldg(q0 + (size_t)i * ld), f1 = __ldg(q1 + (size_t)i * ld), f2 = __ldg(q2 + (size_t)i * ld);
        if (is_zero(w)) continue;
        const double a = f1 - f2, b = f2 - f0, d = f0 - f1;
        D0 = fma(w * a, a, D0);
        D1 = fma(w * b, b, D1);
        D2 = fma(w * d, d, D2);
    }
    const v3 x0 = load(V, c[0]), x1 = load(V, c[1]), x2 = load(V, c[2]);
    const v3 e0 = sub(x2, x1), e1 = sub(x0, x2), e2 = sub(x1, x0);
    const v3 nrm = cross(e1, e2);
    const double s = sqrt(dot(nrm, nrm)), inv = 1.0 / s;
    const double t0 = -dot(e1, e2), t1 = -dot(e2, e0), t2 = -dot(e0, e1);
    const double P = Pv[c[0]] + Pv[c[1]] + Pv[c[2]];
    const double N = fma(t0, D0, fma(t1, D1, t2 * D2));
    const double Es = fma(-0.5 * N * inv, inv, P * (-1.0 / 6.0)), h = 0.5 * inv;
    const v3 C0 = mul(h * (D1 + D2 - D0), e0), C1 = mul(h * (D2 + D0 - D1), e1), C2 = mul(h * (D0 + D1 - D2), e2);
    const v3 ns = mul(Es * inv, nrm);
    const v3 g0 = add(sub(C1, C2), cross(ns, e0)), g1 = add(sub(C2, C0), cross(ns, e1));
    atomic_add3(g, c[0], g0);
    atomic_add3(g, c[1], g1);
    atomic_add3(g, c[2], {-(g0.x + g1.x), -(g0.y + g1.y), -(g0.z + g1.z)});
}

}  // namespace

void eig_grad(cudaStream_t s, int n, int m, int p, const double *V, const int *F, const double *evals,
              const double *evecs, int ld, const double *dloss, double *dV, double *Pv) {
    HSIM_CUDA(cudaMemsetAsync(dV, 0, sizeof(double) * 3 * (size_t)n, s));
    if (m == 0) return;
    k_vertex_energy<<<(unsigned)((n + 63) / 64), 64, 0, s>>>(n, p, evals, evecs, ld, dloss, Pv);
    HSIM_LAUNCHED();
    k_eig_grad<<<(unsigned)((m + 63) / 64), 64, 0, s>>>(m, p, V, F, evecs, ld, dloss, Pv, dV);
    HSIM_LAUNCHED();
}

}  // namespace k
}  // namespace hsim
