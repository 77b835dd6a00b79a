// Online stage of the kinetic slab (Sec. 4.2, Eq. rte_cond_reduced): the block-tridiagonal
// normal equations along the chain of patches, H = P^T P with blocks H_mm and
// E_m = H_{m+1,m}, factored as L_m L_m^T = H_mm - C_{m-1} C_{m-1}^T, C_m = E_m L_m^{-T}, and
// c = argmin |P c - d| by the factor and two refinement steps (corrected semi-normal
// equations), then the reconstruction.
//
// The chain over the patches is the only serial part.  Everything else (the blocks of H,
// residual rows, P^T r, products with L_m^{-1}, the reconstruction) runs over the whole
// GPU, and the chain's triangular solves are turned into one product per patch by
// matrices formed with the factor:
//   forward   y_m = L_m^{-1} g_m - (L_m^{-1} C_{m-1}) y_{m-1},
//   backward  x_m = L_m^{-T} y_m - (L_m^{-T} C_m^T) x_{m+1}.
// As one CTA for the whole factor and one per data set, with the triangular solves on
// one thread, the 8192-cell slab of 64 patches took 44 ms to factor and 124 ms to solve;
// now 7.2 ms of chain, 1.2 of sweeps and 0.6 of the rest.  The smallest slabs keep one CTA
// for the factor's chain, and one per data set for a whole solve.
#include "kinetic_online.h"
#include "device_util.cuh"
#include "patch_dense.h"

#include <algorithm>
#include <cooperative_groups.h>

namespace cg = cooperative_groups;

namespace msp {

namespace {

constexpr int kKfThreads = 512;
constexpr int kKfMaxK = 160;         // largest block the factor holds in shared memory
constexpr int kKfChunk = 8192;       // doubles of C staged at a time

// H_mm (into L) and E_m (into C): 16 x 16 outputs per CTA; blockIdx (tile, patch)
__global__ void __launch_bounds__(256) kinetic_blocks_kernel(KOnArgs A, double* L, double* C) {
    const int nv = A.nv, M = A.M;
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    for (int m = blockIdx.y; m < M; m += gridDim.y) {
        const int km = A.k[m], t = (km + 15) / 16;
        const KPatchDev P = A.patches[m];
        const double* Qm = A.Q + A.q_off[m];
        const int last = P.x1 - P.x0;
        const int nt = t * t;
        if ((int)blockIdx.x < nt) {
            const int i = (blockIdx.x % t) * 16 + tx, j = (blockIdx.x / t) * 16 + ty;
            if (i < km && j < km) {
                double a = 0.0;
                for (int l = 0; l < nv; ++l) {
                    // right-interface rows (m < M-1), left-interface rows (m > 0), incoming rows
                    const bool right = (m < M - 1) || (A.v[l] < 0.0);
                    const bool left = (m > 0) || (A.v[l] > 0.0);
                    if (right)
                        a += Qm[(long long)last * nv + l + (long long)i * P.n_k] *
                             Qm[(long long)last * nv + l + (long long)j * P.n_k];
                    if (left) a += Qm[l + (long long)i * P.n_k] * Qm[l + (long long)j * P.n_k];
                }
                L[A.l_off[m] + i + (long long)j * km] = a;
            }
        }
        if (m + 1 < M) {
            const int kn = A.k[m + 1], tn = (kn + 15) / 16;
            if ((int)blockIdx.x < tn * t) {
                const KPatchDev Pn = A.patches[m + 1];
                const double* Qn = A.Q + A.q_off[m + 1];
                const int i = (blockIdx.x % tn) * 16 + tx, j = (blockIdx.x / tn) * 16 + ty;
                if (i < kn && j < km) {
                    double a = 0.0;
                    for (int l = 0; l < nv; ++l)
                        a -= Qn[l + (long long)i * Pn.n_k] * Qm[(long long)last * nv + l + (long long)j * P.n_k];
                    C[A.cb_off[m] + i + (long long)j * kn] = a;
                }
            }
        }
    }
}

// The chain of the factor on one cluster: per patch the update by C_{m-1} (columns dealt to
// the CTAs), the Cholesky in the first CTA's shared memory (LDL^T form, one barrier per
// column: the thread that makes the last update of the next pivot takes its
// reciprocal), and the rows of C_m by forward substitution, a warp per row.
__global__ void __launch_bounds__(kKfThreads) kinetic_chain_kernel(KOnArgs A, double* Lf, double* Cf, int* fail) {
    extern __shared__ __align__(16) double ksm[];
    __shared__ double s_inv[2];
    __shared__ int s_ok;
    cg::cluster_group cl = cg::this_cluster();
    const int nc = (int)cl.num_blocks(), rank = (int)cl.block_rank();
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = blockDim.x >> 5;
    if (tid == 0) s_ok = 1;
    for (int m = 0; m < A.M; ++m) {
        const int km = A.k[m];
        double* D = Lf + A.l_off[m];
        if (m > 0 && km > 0) {                           // D -= C_{m-1} C_{m-1}^T, lower triangle
            const int kp = A.k[m - 1];
            const double* Cp = Cf + A.cb_off[m - 1];
            const int qc = max(1, kKfChunk / km);
            // column j = rank + nc (warp + nw u) of this CTA, rows j + lane, ...
            for (int q0 = 0; q0 < kp; q0 += qc) {
                const int qn = min(qc, kp - q0);
                __syncthreads();
                for (int e = tid; e < qn * km; e += blockDim.x) ksm[e] = __ldcg(Cp + (long long)q0 * km + e);
                __syncthreads();
                for (int j = rank + nc * warp; j < km; j += nc * nw)
                    for (int i = j + lane; i < km; i += 32) {
                        double a = 0.0;
                        for (int q = 0; q < qn; ++q) a += ksm[q * km + i] * ksm[q * km + j];
                        double* d = D + i + (long long)j * km;
                        __stcg(d, __ldcg(d) - a);
                    }
            }
            __threadfence();
        }
        cl.sync();
        const int ld = km | 1;                           // row-major in shared memory: L[i][j] at i ld + j
        if (rank == 0 && km > 0) {
            for (int e = tid; e < km * km; e += blockDim.x) {
                const int i = e % km, j = e / km;
                if (i >= j) ksm[i * ld + j] = __ldcg(D + e);
            }
            __syncthreads();
            auto pivot = [&](double d) {
                if (!(d > 0.0)) {
                    s_ok = 0;
                    return 1.0;
                }
                return d;
            };
            if (tid == 0) {
                const double d = pivot(ksm[0]);
                ksm[0] = d;
                s_inv[0] = 1.0 / d;
            }
            __syncthreads();
            const int rp = (km + 31) / 32 * 32, G = max(1, (int)blockDim.x / rp);
            const int ri = tid % rp, g = tid / rp;
            for (int k = 0; k < km; ++k) {
                if (g < G && ri > k && ri < km) {
                    const double t = ksm[ri * ld + k] * s_inv[k & 1];
                    for (int j = k + 1 + g; j <= ri; j += G) ksm[ri * ld + j] = fma(-t, ksm[j * ld + k], ksm[ri * ld + j]);
                    if (g == 0 && ri == k + 1) {         // the next pivot is final
                        const double d = pivot(ksm[ri * ld + ri]);
                        ksm[ri * ld + ri] = d;
                        s_inv[(k + 1) & 1] = 1.0 / d;
                    }
                }
                __syncthreads();
            }
            for (int e = tid; e < km * km; e += blockDim.x) {
                const int i = e % km, j = e / km;
                const double sq = sqrt(ksm[j * ld + j]);
                __stcg(D + e, i > j ? ksm[i * ld + j] / sq : (i == j ? sq : 0.0));
            }
            __threadfence();
        }
        cl.sync();
        if (m + 1 < A.M && km > 0) {                     // rows of C_m = E_m L_m^{-T}
            const int kn = A.k[m + 1];
            double* Cm = Cf + A.cb_off[m];
            // columns of L contiguous, L[i][j] at j ld + i (conflict-free along the lanes), with
            // the reciprocals of the diagonal in its place
            for (int e = tid; e < km * km; e += blockDim.x) {
                const int i = e % km, j = e / km;
                if (i >= j) ksm[j * ld + i] = i == j ? 1.0 / __ldcg(D + e) : __ldcg(D + e);
            }
            __syncthreads();
            constexpr int kR = kKfMaxK / 32;
            for (int r = rank + nc * warp; r < kn; r += nc * nw) {
                double x[kR];
#pragma unroll
                for (int u = 0; u < kR; ++u) x[u] = lane + 32 * u < km ? __ldcg(Cm + r + (long long)(lane + 32 * u) * kn) : 0.0;
                for (int j = 0; j < km; ++j) {
                    double v = 0.0;
#pragma unroll
                    for (int u = 0; u < kR; ++u)
                        if (u == j >> 5) v = x[u];
                    v = __shfl_sync(0xffffffffu, v, j & 31) * ksm[j * ld + j];
#pragma unroll
                    for (int u = 0; u < kR; ++u) {
                        const int l = lane + 32 * u;
                        if (l == j) x[u] = v;
                        else if (l > j && l < km) x[u] = fma(-ksm[j * ld + l], v, x[u]);
                    }
                }
#pragma unroll
                for (int u = 0; u < kR; ++u)
                    if (lane + 32 * u < km) __stcg(Cm + r + (long long)(lane + 32 * u) * kn, x[u]);
            }
            __threadfence();
        }
        cl.sync();
    }
    if (rank == 0 && tid == 0) *fail = s_ok ? 0 : 1;
}

// The chain on one CTA out of global memory, for blocks beyond kKfMaxK and for the smallest
__global__ void __launch_bounds__(kKfThreads) kinetic_chain_global_kernel(KOnArgs A, double* Lf, double* Cf, int* fail) {
    __shared__ int s_ok;
    if (threadIdx.x == 0) s_ok = 1;
    __syncthreads();
    for (int m = 0; m < A.M; ++m) {
        const int km = A.k[m];
        double* D = Lf + A.l_off[m];
        if (m > 0) {
            const int kp = A.k[m - 1];
            const double* Cp = Cf + A.cb_off[m - 1];
            for (int e = threadIdx.x; e < km * km; e += blockDim.x) {
                const int i = e % km, j = e / km;
                if (i < j) continue;
                double a = 0.0;
                for (int q = 0; q < kp; ++q) a += Cp[i + (long long)q * km] * Cp[j + (long long)q * km];
                D[e] -= a;
            }
            __syncthreads();
        }
        for (int c = 0; c < km; ++c) {
            if (threadIdx.x == 0) {
                const double d = D[c + (long long)c * km];
                if (!(d > 0.0)) { s_ok = 0; D[c + (long long)c * km] = 1.0; }
                else D[c + (long long)c * km] = sqrt(d);
            }
            __syncthreads();
            const double piv = D[c + (long long)c * km];
            for (int i = c + 1 + threadIdx.x; i < km; i += blockDim.x) D[i + (long long)c * km] /= piv;
            __syncthreads();
            const int R = km - c - 1;
            for (int e = threadIdx.x; e < R * R; e += blockDim.x) {
                const int i = c + 1 + e % R, j = c + 1 + e / R;
                if (i >= j) D[i + (long long)j * km] -= D[i + (long long)c * km] * D[j + (long long)c * km];
            }
            __syncthreads();
        }
        for (int e = threadIdx.x; e < km * km; e += blockDim.x)
            if (e % km < e / km) D[e] = 0.0;
        __syncthreads();
        if (m + 1 < A.M) {
            const int kn = A.k[m + 1];
            double* Cm = Cf + A.cb_off[m];
            for (int i = threadIdx.x; i < kn; i += blockDim.x)
                for (int j = 0; j < km; ++j) {           // forward substitution on row i
                    double a = Cm[i + (long long)j * kn];
                    for (int q = 0; q < j; ++q) a -= D[j + (long long)q * km] * Cm[i + (long long)q * kn];
                    Cm[i + (long long)j * kn] = a / D[j + (long long)j * km];
                }
            __syncthreads();
        }
    }
    if (threadIdx.x == 0) *fail = s_ok ? 0 : 1;
}

// ------------------------------------------------------------------ solve
// Work of data set b: c, g, t (Np each), r (rows).  Row layout: interface m (m < M-1): nv
// rows; then nv/2 left incoming rows (positive v, ascending), then nv/2 right incoming rows.
struct KVec {
    double* base;
    long long stride;
    int Np;
    __device__ double* c(int b) const { return base + b * stride; }
    __device__ double* g(int b) const { return c(b) + Np; }
    __device__ double* t(int b) const { return c(b) + 2LL * Np; }
    __device__ double* r(int b) const { return c(b) + 3LL * Np; }
};

// value of u_m at node `node`, velocity l for coefficients c_m
__device__ __forceinline__ double kval(const KOnArgs& A, int m, int node, int l, const double* c) {
    const long long n_k = A.patches[m].n_k;
    const double* Qm = A.Q + A.q_off[m] + (long long)node * A.nv + l;
    const double* cm = c + A.c_off[m];
    const int km = A.k[m];
    double a = 0.0;
#pragma unroll 8
    for (int j = 0; j < km; ++j) a += Qm[j * n_k] * cm[j];
    return a;
}

// residual rows r = d - P c (c = 0 on the first pass): rows t0, t0 + step, ... of data set b
__device__ __forceinline__ void residual_rows(const KOnArgs& A, const KVec& W, const double* inflow, int first, int b,
                                              int t0, int step) {
    const int nv = A.nv, M = A.M, rows = M * nv;
    const double* inl = inflow + (long long)b * 2 * nv;
    const double* inr = inl + nv;
    const double* c = W.c(b);
    for (int t = t0; t < rows; t += step) {
        double v;
        if (t < (M - 1) * nv) {
            const int m = t / nv, l = t - m * nv, last = A.patches[m].x1 - A.patches[m].x0;
            v = first ? 0.0 : -(kval(A, m, last, l, c) - kval(A, m + 1, 0, l, c));
        } else if (t < (M - 1) * nv + nv / 2) {
            const int l = nv / 2 + t - (M - 1) * nv;
            v = inl[l] - (first ? 0.0 : kval(A, 0, 0, l, c));
        } else {
            const int l = t - (M - 1) * nv - nv / 2, last = A.patches[M - 1].x1 - A.patches[M - 1].x0;
            v = inr[l] - (first ? 0.0 : kval(A, M - 1, last, l, c));
        }
        W.r(b)[t] = v;
    }
}

// g = P^T r, then t = L^{-1} g: patches m0, m0 + step, ... of data set b, g in gs
__device__ __forceinline__ void rhs_patches(const KOnArgs& A, const KVec& W, int b, int m0, int step, double* gs) {
    const int nv = A.nv, M = A.M, lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const double* r = W.r(b);
    for (int m = m0; m < M; m += step) {
        const KPatchDev P = A.patches[m];
        const int km = A.k[m], last = P.x1 - P.x0;
        for (int j = warp; j < km; j += nw) {
            const double* q0 = A.Q + A.q_off[m] + (long long)j * P.n_k;
            const double* q1 = q0 + (long long)last * nv;
            double a = 0.0;
            for (int l = lane; l < nv; l += 32) {
                if (m < M - 1) a += q1[l] * r[m * nv + l];
                else if (l < nv / 2) a += q1[l] * r[(M - 1) * nv + nv / 2 + l];
                if (m > 0) a -= q0[l] * r[(m - 1) * nv + l];
                else if (l >= nv / 2) a += q0[l] * r[(M - 1) * nv + l - nv / 2];
            }
            a = warp_sum(a);
            if (lane == 0) gs[j] = a;
        }
        __syncthreads();
        const double* Fi = A.Fi + A.l_off[m];            // L^{-T}: column i holds row i of L^{-1}
        for (int i = warp; i < km; i += nw) {
            double a = 0.0;
            for (int q = lane; q <= i; q += 32) a += Fi[q + (long long)i * km] * gs[q];
            a = warp_sum(a);
            if (lane == 0) W.t(b)[A.c_off[m] + i] = a;
        }
        __syncthreads();
    }
}

// w = L^{-T} y (y in t, w into g): patches m0, m0 + step, ... of data set b, y in ys
__device__ __forceinline__ void lit_patches(const KOnArgs& A, const KVec& W, int b, int m0, int step, double* ys) {
    for (int m = m0; m < A.M; m += step) {
        const int km = A.k[m];
        const double* Fi = A.Fi + A.l_off[m];
        for (int i = threadIdx.x; i < km; i += blockDim.x) ys[i] = W.t(b)[A.c_off[m] + i];
        __syncthreads();
        for (int i = threadIdx.x; i < km; i += blockDim.x) {
            double a = 0.0;
#pragma unroll 8
            for (int q = i; q < km; ++q) a += Fi[i + (long long)q * km] * ys[q];
            W.g(b)[A.c_off[m] + i] = a;
        }
        __syncthreads();
    }
}

// One chain: z_m = s_m - T_m z_{m -+ 1} along the patches (T_m: k_m x k_{m -+ 1}), one CTA of
// kKfThreads per data set; the rows' sums are split over the threads that share a row.  The
// next patch's matrix is brought into the L2 meanwhile.  Forward: in place in t.
// Backward: s in g, and c += z.  zs: z of two patches, partial sums.
__device__ __forceinline__ void chain_sweep(const KOnArgs& A, const KVec& W, int b, int backward, double* zs) {
    const int tid = threadIdx.x, M = A.M;
    const int kx = A.k_max;
    double* part = zs + 2 * kx;                          // kKfThreads
    double* src = backward ? W.g(b) : W.t(b);
    double* c = W.c(b);
    const double* T = backward ? A.Tb : A.Tf;
    for (int s = 0; s < M; ++s) {
        const int m = backward ? M - 1 - s : s, km = A.k[m];
        const int mp = backward ? m + 1 : m - 1, kp = s > 0 ? A.k[mp] : 0;
        double* z = zs + (s & 1) * kx;
        const double* zp = zs + ((s + 1) & 1) * kx;
        const double* Tm = s > 0 ? T + A.cb_off[backward ? m : m - 1] : nullptr;
        if (s + 1 < M) {
            const int mn = backward ? m - 1 : m + 1;
            const double* Tn = T + A.cb_off[backward ? mn : m];
            const long long n = (long long)A.k[mn] * km;
            for (long long e = 16LL * tid; e < n; e += 16LL * kKfThreads) asm volatile("prefetch.global.L2 [%0];" ::"l"(Tn + e));
        }
        const int rows = (km + 31) / 32 * 32;            // beyond kKfThreads rows: one part, several rounds
        const int parts = rows > 0 ? max(1, kKfThreads / rows) : 1;
        const int p = rows > 0 ? tid / rows : 0;
        for (int i0 = 0; i0 < km; i0 += kKfThreads) {
            const int i = i0 + (rows > 0 ? tid % rows : 0);
            double a = 0.0;
            if (i < km && p < parts) {
#pragma unroll 4
                for (int q = p; q < kp; q += parts) a += Tm[i + (long long)q * km] * zp[q];
            }
            part[tid] = a;
            __syncthreads();
            if (p == 0 && i < km) {
                for (int u = 1; u < parts; ++u) a += part[tid + u * rows];
                const double v = src[A.c_off[m] + i] - a;
                z[i] = v;
                if (backward) c[A.c_off[m] + i] += v;
                else src[A.c_off[m] + i] = v;
            }
            __syncthreads();
        }
    }
}

// reconstruction: patch interiors, interface averages, incoming data at the ends; values
// (node, velocity) t0, t0 + step, ... of data set b
__device__ __forceinline__ void recon_values(const KOnArgs& A, const KVec& W, const double* inflow, double* f_out,
                                             double* c_out, int b, long long t0, long long step) {
    const int nv = A.nv, M = A.M, N = A.N;
    const double* inl = inflow + (long long)b * 2 * nv;
    const double* inr = inl + nv;
    const double* c = W.c(b);
    const long long total = (long long)(N + 1) * nv;
    const int Wd = A.patches[0].x1 - A.patches[0].x0;
    for (long long t = t0; t < total; t += step) {
        const int i = (int)(t / nv), l = (int)(t % nv);
        const int m = min(i / Wd, M - 1);
        double val;
        if (i == A.patches[m].x0 && m > 0)
            val = 0.5 * (kval(A, m - 1, A.patches[m - 1].x1 - A.patches[m - 1].x0, l, c) + kval(A, m, 0, l, c));
        else
            val = kval(A, m, i - A.patches[m].x0, l, c);
        if (i == 0 && A.v[l] > 0.0) val = inl[l];
        if (i == N && A.v[l] < 0.0) val = inr[l];
        f_out[b * total + t] = val;
    }
    if (c_out)
        for (long long j = t0; j < W.Np; j += step) c_out[(long long)b * W.Np + j] = c[j];
}

// The phases by themselves: blockIdx (data set, tile or patch)
__global__ void __launch_bounds__(128) kinetic_residual_kernel(KOnArgs A, KVec W, const double* inflow, int first) {
    residual_rows(A, W, inflow, first, blockIdx.x, blockIdx.y * 128 + threadIdx.x, 128 * gridDim.y);
}
__global__ void __launch_bounds__(256) kinetic_rhs_kernel(KOnArgs A, KVec W) {
    extern __shared__ double ksv[];
    rhs_patches(A, W, blockIdx.x, blockIdx.y, gridDim.y, ksv);
}
__global__ void __launch_bounds__(kKfThreads) kinetic_sweep_kernel(KOnArgs A, KVec W, int backward) {
    extern __shared__ double ksv[];
    chain_sweep(A, W, blockIdx.x, backward, ksv);
}
__global__ void __launch_bounds__(256) kinetic_lit_kernel(KOnArgs A, KVec W) {
    extern __shared__ double ksv[];
    lit_patches(A, W, blockIdx.x, blockIdx.y, gridDim.y, ksv);
}
__global__ void __launch_bounds__(256) kinetic_recon_kernel(KOnArgs A, KVec W, const double* inflow, double* f_out,
                                                            double* c_out) {
    recon_values(A, W, inflow, f_out, c_out, blockIdx.x, blockIdx.y * 256LL + threadIdx.x, 256LL * gridDim.y);
}

// All of them, one CTA per data set, for slabs so small that sixteen launches take longer
// than the work
__global__ void __launch_bounds__(kKfThreads) kinetic_small_kernel(KOnArgs A, KVec W, const double* inflow, double* f_out,
                                                                   double* c_out) {
    extern __shared__ double ksv[];
    const int b = blockIdx.x;
    for (int pass = 0; pass < 3; ++pass) {
        residual_rows(A, W, inflow, pass == 0, b, threadIdx.x, blockDim.x);
        __syncthreads();
        rhs_patches(A, W, b, 0, 1, ksv);
        chain_sweep(A, W, b, 0, ksv);
        __syncthreads();
        lit_patches(A, W, b, 0, 1, ksv);
        chain_sweep(A, W, b, 1, ksv);
        __syncthreads();
    }
    recon_values(A, W, inflow, f_out, c_out, b, threadIdx.x, blockDim.x);
}

}  // namespace

msp_status kinetic_factor(const KOnArgs& A, const std::vector<int>& k, const std::vector<long long>& l_off,
                          const std::vector<long long>& cb_off, double* Lf, double* Cf, double* Fi, double* Tf, double* Tb,
                          int* failed, cudaStream_t s) {
    const int M = A.M;
    const int t = (A.k_max + 15) / 16;
    if (A.k_max > 0) {
        kinetic_blocks_kernel<<<dim3(t * t, std::min(M, 65535)), 256, 0, s>>>(A, Lf, Cf);
        count_launches(1);
    }
    DevBuf<int> fail;
    MSP_TRY(fail.alloc(1, s));
    // Below eight columns a block's barriers on a cluster take longer than its work by one CTA: 1024
    // patches of 2 or 4 columns 6.9 and 8.7 ms against 3.4 and 6.4 (256 of 8: 3.06 against 3.36)
    if (A.k_max >= 8 && A.k_max <= kKfMaxK) {
        const size_t smem = sizeof(double) * std::max<size_t>((size_t)A.k_max * (A.k_max | 1), kKfChunk + A.k_max);
        MSP_TRY(allow_smem(kinetic_chain_kernel, smem));
        cudaLaunchConfig_t cfg{};
        cfg.gridDim = dim3(kPatchCluster);
        cfg.blockDim = dim3(kKfThreads);
        cfg.dynamicSmemBytes = smem;
        cfg.stream = s;
        cudaLaunchAttribute at{};
        at.id = cudaLaunchAttributeClusterDimension;
        at.val.clusterDim.x = kPatchCluster;
        at.val.clusterDim.y = at.val.clusterDim.z = 1;
        cfg.attrs = &at;
        cfg.numAttrs = 1;
        MSP_CUDA(cudaLaunchKernelEx(&cfg, kinetic_chain_kernel, A, Lf, Cf, fail.p));
    } else {
        kinetic_chain_global_kernel<<<1, kKfThreads, 0, s>>>(A, Lf, Cf, fail.p);
    }
    count_launches(1);
    MSP_CUDA(cudaGetLastError());
    MSP_CUDA(cudaMemcpyAsync(failed, fail.p, sizeof(int), cudaMemcpyDeviceToHost, s));
    MSP_CUDA(cudaStreamSynchronize(s));
    if (*failed) return MSP_OK;
    // L^{-T}, and the chains' matrices L_{m+1}^{-1} C_m and L_m^{-T} C_m^T
    const PatchClasses classes = classify_patches(k, l_off);
    DevBuf<PatchBlock> blocks;
    MSP_TRY(upload(blocks, classes.blocks, s));
    MSP_TRY(patch_triangular_inverse(classes, blocks.p, Lf, Fi, s));
    std::vector<GemmDesc> gf, gb;
    int kmax = 1;
    for (int m = 0; m + 1 < M; ++m) {
        if (k[m] == 0 || k[m + 1] == 0) continue;
        gf.push_back(GemmDesc{Fi + l_off[m + 1], Cf + cb_off[m], Tf + cb_off[m], k[m + 1], k[m], k[m + 1], k[m + 1],
                              k[m + 1], k[m + 1], 1.0, 0.0});
        gf.back().a_lower = 1;                           // op(A) = L^{-1}
        gb.push_back(GemmDesc{Fi + l_off[m], Cf + cb_off[m], Tb + cb_off[m], k[m], k[m + 1], k[m], k[m], k[m + 1], k[m],
                              1.0, 0.0});
        kmax = std::max(kmax, std::max(k[m], k[m + 1]));
    }
    DevBuf<GemmDesc> d_gf, d_gb;
    MSP_TRY(upload(d_gf, gf, s));
    MSP_TRY(upload(d_gb, gb, s));
    gemm_batched<double>(d_gf.p, (int)gf.size(), kmax, kmax, true, false, s, kGemmStructured);
    gemm_batched<double>(d_gb.p, (int)gb.size(), kmax, kmax, false, true, s);
    MSP_CUDA(cudaGetLastError());
    MSP_CUDA(cudaStreamSynchronize(s));   // the tables above are released on return
    return MSP_OK;
}

// One launch in place of sixteen: up to 64 columns over the patches and 2^17 terms of the
// reconstruction.  A call for one data set, one launch against sixteen: 1 patch of 2 columns 54 us
// against 107, 3 of 2 85 against 134, 4 of 16 138 against 171, 8 of 8 183 against 191; beyond it
// 16 of 8 326 against 289, 4 of 32 250 against 192; 4 of 8 with 2049 nodes (2^17 terms) 152
// against 154.
static bool small_slab(const KOnArgs& A) {
    return (long long)A.M * A.k_max <= 64 && (long long)(A.N + 1) * A.nv * std::max(A.k_max, 1) <= 1 << 17;
}

msp_status kinetic_online(const KOnArgs& A, int Np, const double* inflow, int batch, double* f_out, double* c_out,
                          cudaStream_t s) {
    const int M = A.M, nv = A.nv, n1 = std::max(Np, 1);
    DevBuf<double> work;
    KVec W{};
    W.Np = n1;
    W.stride = 3LL * n1 + (long long)M * nv;
    MSP_TRY(work.alloc((size_t)batch * W.stride, s));
    W.base = work.p;
    MSP_CUDA(cudaMemsetAsync(work.p, 0, sizeof(double) * (size_t)batch * W.stride, s));
    const size_t vec = sizeof(double) * std::max(A.k_max, 1);
    const size_t chain = 2 * vec + sizeof(double) * kKfThreads;
    const unsigned pm = (unsigned)std::min(M, 65535);
    const long long total = (long long)(A.N + 1) * nv;
    if (small_slab(A)) {
        kinetic_small_kernel<<<batch, kKfThreads, chain, s>>>(A, W, inflow, f_out, c_out);
        count_launches(1);
        MSP_CUDA(cudaGetLastError());
        MSP_CUDA(cudaStreamSynchronize(s));   // the work buffer is released on return
        return MSP_OK;
    }
    for (int pass = 0; pass < 3; ++pass) {
        kinetic_residual_kernel<<<dim3(batch, std::min(1024, (M * nv + 127) / 128)), 128, 0, s>>>(A, W, inflow, pass == 0);
        kinetic_rhs_kernel<<<dim3(batch, pm), 256, vec, s>>>(A, W);
        kinetic_sweep_kernel<<<batch, kKfThreads, chain, s>>>(A, W, 0);
        kinetic_lit_kernel<<<dim3(batch, pm), 256, vec, s>>>(A, W);
        kinetic_sweep_kernel<<<batch, kKfThreads, chain, s>>>(A, W, 1);
        count_launches(5);
    }
    kinetic_recon_kernel<<<dim3(batch, (unsigned)std::min<long long>(16384, (total + 255) / 256)), 256, 0, s>>>(
        A, W, inflow, f_out, c_out);
    count_launches(1);
    MSP_CUDA(cudaGetLastError());
    MSP_CUDA(cudaStreamSynchronize(s));   // the work buffer is released on return
    return MSP_OK;
}

}  // namespace msp
