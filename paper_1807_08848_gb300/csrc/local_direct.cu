// Direct batched local solves: the local solver of Algorithm alg:summary
// (LocalPDESolver on every buffered patch, Eq. elliptic_random for the ring
// data) as a factorisation of each patch's operator that every column of the
// patch shares, in place of an iteration per column.  The paper allows any
// standard local solver; this one is a block LDL^T over the grid rows.
//
// Scaled operator A~ = S A S, S = diag(A)^(-1/2), on the interior nx x ny nodes:
// block tridiagonal over the rows j = 0..ny-1, diagonal blocks T_j (tridiagonal,
// unit diagonal, off-diagonal -a_E s s), couplings -diag(c_j) between rows j and
// j+1 with c_j[i] = a_N(i, j+1/2) s_j[i] s_{j+1}[i].
//   Factorisation (FP32):  Z_0 = T_0,  Z_j = T_j - C_{j-1} W_{j-1} C_{j-1},
//                          W_j = Z_j^{-1}  (Gauss-Jordan; Z_j is SPD).
//   Solve A~ d = g:        forward  y_0 = g_0,  w_j = W_j y_j,  y_{j+1} = g_{j+1} + c_j o w_j;
//                          backward d_{ny-1} = w_{ny-1},  d_j = w_j + W_j (c_j o d_{j+1}).
// Every step of both sweeps is a product of the nx x nx block W_j with an nx x 64 or
// nx x 32 block of columns, so the sweeps are dense contractions that a CTA runs out of
// shared memory.
// Accuracy comes from FP64 iterative refinement: r = b - A x in FP64 (b from
// the ring data: x holds the ring values), g = S r rounded to FP32, x += S d,
// until |r| <= tol |b| per column (a few passes: the FP32 factor reduces the
// residual by about 1e-5 per pass on the workloads' media).
//
// Storage (per patch, offsets in the Direct tables):
//   W  ny x ld x ld floats (ld = nx rounded up to 4, zero padding), W_j(i, k) at
//      [k / 4][i][k mod 4]: four terms of a row are one 16-byte load
//   s  ny x nx doubles; D  ny x nx floats (row j: c_j, zero on the last row)
//   X  cols x (ny+2) x (nx+2) doubles: the FP64 iterate with its ring values
//   R  chunks x ny x 32 x nx floats: the scaled residual g, column-major per row
//   K  chunks x ny x 32 x ld floats: the forward sweep's w_j, a column's row contiguous
#include "internal.h"
#include "device_util.cuh"

#include <algorithm>
#include <vector>

namespace msp {

namespace {

constexpr int kDirThreads = 256;
constexpr int kCB = 32;          // columns per chunk
constexpr int kDirMaxLd = 160;   // widest padded interior row handled (5 groups of 32 rows)
constexpr int kDirMaxPasses = 8; // refinement passes at most

struct DirArgs {
    int N;
    const double* aE;
    const double* aN;
    const PatchDev* patches;
    const int* bpos;
    uint64_t seed;
    const long long *w_off, *s_off, *x_off, *r_off, *k_off;
    const int* col_base;
    const int2* cols;
    const int4* chunks;
    const int4* ctas;
    const int* stat_idx;
    float* W;
    float* D;
    float* R;
    float* K;
    double* s;
    double* X;
    double* b2;
    double* r2;
    int* active;
    int* passes;
    double* snaps;
    int* stats;
    double tol;
    int patch0, col0;          // first patch and column of the launch's group
};

struct Geo {
    int nx, ny, wd, hd, ld;
};

__host__ __device__ inline Geo geo(const PatchDev& P) {
    Geo g;
    g.nx = P.X1 - P.X0 - 1;
    g.ny = P.Y1 - P.Y0 - 1;
    g.wd = g.nx + 2;
    g.hd = g.ny + 2;
    g.ld = g.nx > 0 ? (g.nx + 3) / 4 * 4 : 0;
    return g;
}

// ------------------------------------------------------------------ factor
// One CTA per patch: s, the couplings c_j, and W_j = Z_j^{-1} row by row.  The
// block lives in registers: thread (tr, tc) of a 16 x 16 layout holds the TS x TS
// sub-block of rows tr TS .., columns tc TS .. (TS = ceil(ld / 16), one value for the
// launch).  Z_j = T_j - C_{j-1} W_{j-1} C_{j-1} is formed elementwise from the
// registers holding W_{j-1}; Gauss-Jordan inversion in place without pivoting (Z_j
// is SPD), TS pivots at a time: the thread of the diagonal sub-block runs its own pivots
// and publishes the multipliers, the threads of its rows and columns apply them to
// theirs and publish the pivot rows and column multipliers, all others apply the TS
// rank-one updates out of shared memory -- two barriers for TS pivots, every element the
// same operations in the same order as one pivot at a time.  W_j goes to global memory
// through a padded shared copy (coalesced stores).  Bound: the latency of the pivot
// chain, one CTA per patch.  One pivot per barrier took 50 ms on 1024 patches of 95
// interior nodes a row, now 18.
template <int TS>
__global__ void __launch_bounds__(kDirThreads) direct_factor_kernel(DirArgs A) {
    extern __shared__ __align__(16) float fsm[];
    const int m = A.patch0 + blockIdx.x;
    const PatchDev P = A.patches[m];
    const Geo g = geo(P);
    if (g.nx < 1 || g.ny < 1) return;
    const int n = g.nx, ld = g.ld, N = A.N;
    constexpr int kW = 16 * TS;    // rows (and columns) the thread layout covers
    float* Zs = fsm;               // ld x (ld + 1): staging of W_j for the transposed store
    float* RK = Zs + ld * (ld + 1);   // TS x kW: pivot rows before their scaling
    float* FR = RK + TS * kW;         // TS x kW: column multipliers
    __shared__ float s_inv[TS], s_fr[TS][TS], s_rk[TS][TS];   // diagonal sub-block: 1 / pivot, multipliers, rows
    double* sv = A.s + A.s_off[m];
    float* Dv = A.D + A.s_off[m];
    float* Wout = A.W + A.w_off[m];
    const double* aE = A.aE;
    const double* aN = A.aN;
    for (int t = threadIdx.x; t < n * g.ny; t += blockDim.x) {
        const int j = t / n, i = t - j * n;
        const long long gi = P.X0 + 1 + i, gj = P.Y0 + 1 + j;
        const double d = aE[gj * N + gi - 1] + aE[gj * N + gi] + aN[(gj - 1) * (N + 1) + gi] + aN[gj * (N + 1) + gi];
        sv[t] = 1.0 / sqrt(d);
    }
    __syncthreads();
    for (int t = threadIdx.x; t < n * g.ny; t += blockDim.x) {
        const int j = t / n, i = t - j * n;
        float c = 0.f;
        if (j + 1 < g.ny) {
            const long long gi = P.X0 + 1 + i, gj = P.Y0 + 1 + j;
            c = (float)(aN[gj * (N + 1) + gi] * sv[t] * sv[t + n]);
        }
        Dv[t] = c;
    }
    __syncthreads();
    const int r0 = (threadIdx.x >> 4) * TS, c0 = (threadIdx.x & 15) * TS;
    float z[TS][TS];
#pragma unroll
    for (int a = 0; a < TS; ++a)
#pragma unroll
        for (int b = 0; b < TS; ++b) z[a][b] = 0.f;
    for (int j = 0; j < g.ny; ++j) {
        const long long gj = P.Y0 + 1 + j;
        // Z_j from T_j and the registers holding W_{j-1}; identity on the padding
#pragma unroll
        for (int a = 0; a < TS; ++a) {
            const int r = r0 + a;
            const float dr = (j > 0 && r < n) ? Dv[(j - 1) * n + r] : 0.f;
#pragma unroll
            for (int b = 0; b < TS; ++b) {
                const int c = c0 + b;
                float v = (r == c) ? 1.f : 0.f;
                if (r < n && c < n) {
                    if (c == r + 1 || c + 1 == r) {
                        const int i = min(r, c);
                        v = -(float)(aE[gj * N + P.X0 + 1 + i] * sv[j * n + i] * sv[j * n + i + 1]);
                    }
                    if (j > 0) v -= dr * z[a][b] * Dv[(j - 1) * n + c];
                }
                z[a][b] = v;
            }
        }
        const int tr = threadIdx.x >> 4, tc = threadIdx.x & 15;
        for (int kb = 0; kb * TS < n; ++kb) {
            const int nb = min(TS, n - kb * TS);
            if (tr == kb && tc == kb) {
#pragma unroll
                for (int k = 0; k < TS; ++k) {
                    if (k >= nb) break;
                    const float inv = 1.f / z[k][k];
                    s_inv[k] = inv;
                    float rk[TS];
#pragma unroll
                    for (int b = 0; b < TS; ++b) {
                        rk[b] = z[k][b];
                        s_rk[k][b] = rk[b];
                    }
#pragma unroll
                    for (int a = 0; a < TS; ++a) {
                        if (a == k) continue;
                        const float fr = z[a][k] * inv;
                        s_fr[k][a] = fr;
#pragma unroll
                        for (int b = 0; b < TS; ++b)
                            if (b != k) z[a][b] = fmaf(-fr, rk[b], z[a][b]);
                        z[a][k] = -fr;
                    }
#pragma unroll
                    for (int b = 0; b < TS; ++b) z[k][b] = b == k ? inv : rk[b] * inv;
                }
            }
            __syncthreads();
            if (tc == kb && tr != kb) {
#pragma unroll
                for (int k = 0; k < TS; ++k) {
                    if (k >= nb) break;
                    const float inv = s_inv[k];
#pragma unroll
                    for (int a = 0; a < TS; ++a) {
                        const float fr = z[a][k] * inv;
                        FR[k * kW + r0 + a] = fr;
#pragma unroll
                        for (int b = 0; b < TS; ++b)
                            if (b != k) z[a][b] = fmaf(-fr, s_rk[k][b], z[a][b]);
                        z[a][k] = -fr;
                    }
                }
            } else if (tr == kb && tc != kb) {
#pragma unroll
                for (int k = 0; k < TS; ++k) {
                    if (k >= nb) break;
                    const float inv = s_inv[k];
#pragma unroll
                    for (int b = 0; b < TS; ++b) {
                        const float rk = z[k][b];
                        RK[k * kW + c0 + b] = rk;
#pragma unroll
                        for (int a = 0; a < TS; ++a)
                            if (a != k) z[a][b] = fmaf(-s_fr[k][a], rk, z[a][b]);
                        z[k][b] = rk * inv;
                    }
                }
            }
            __syncthreads();
            if (tr != kb && tc != kb) {
#pragma unroll
                for (int k = 0; k < TS; ++k) {
                    if (k >= nb) break;
                    float fr[TS], rk[TS];
#pragma unroll
                    for (int a = 0; a < TS; ++a) fr[a] = FR[k * kW + r0 + a];
#pragma unroll
                    for (int b = 0; b < TS; ++b) rk[b] = RK[k * kW + c0 + b];
#pragma unroll
                    for (int a = 0; a < TS; ++a)
#pragma unroll
                        for (int b = 0; b < TS; ++b) z[a][b] = fmaf(-fr[a], rk[b], z[a][b]);
                }
            }
        }
        __syncthreads();
        // W_j to global (padding zero) through the padded shared copy
#pragma unroll
        for (int a = 0; a < TS; ++a)
#pragma unroll
            for (int b = 0; b < TS; ++b) {
                const int r = r0 + a, c = c0 + b;
                if (r < ld && c < ld) Zs[r * (ld + 1) + c] = (r < n && c < n) ? z[a][b] : 0.f;
            }
        __syncthreads();
        float* wj = Wout + (long long)j * ld * ld;
        for (int t = threadIdx.x; t < ld * ld; t += blockDim.x) {
            const int k4 = t / (4 * ld), i = (t >> 2) - k4 * ld;
            wj[t] = Zs[i * (ld + 1) + 4 * k4 + (t & 3)];
        }
        __syncthreads();
    }
}

// ------------------------------------------------------------------ init
// One CTA per column: the FP64 iterate is the ring data with a zero interior.
__global__ void __launch_bounds__(kDirThreads) direct_init_kernel(DirArgs A) {
    const int gcol = A.col0 + blockIdx.x;
    const int2 mc = A.cols[gcol];
    const int m = mc.x, col = mc.y;
    const PatchDev P = A.patches[m];
    const Geo g = geo(P);
    double* x = A.X + A.x_off[m] + (long long)col * g.hd * g.wd;
    for (int t = threadIdx.x; t < g.hd * g.wd; t += blockDim.x) x[t] = 0.0;
    __syncthreads();
    if (col < P.samples) {
        const int npairs = (P.n_ring + 1) >> 1;
        for (int q = threadIdx.x; q < npairs; q += blockDim.x) {
            const double2 z = gaussian_pair(A.seed, (uint32_t)q, (uint32_t)col, (uint32_t)m, kTagElliptic);
            int i, j;
            ring_node(P.X0, P.X1, P.Y0, P.Y1, 2 * q, i, j);
            x[(j - P.Y0) * g.wd + (i - P.X0)] = z.x;
            if (2 * q + 1 < P.n_ring) {
                ring_node(P.X0, P.X1, P.Y0, P.Y1, 2 * q + 1, i, j);
                x[(j - P.Y0) * g.wd + (i - P.X0)] = z.y;
            }
        }
    } else if (threadIdx.x == 0) {
        const int t0 = A.bpos[P.bpos_offset + (col - P.samples)];
        int i, j;
        ring_node(P.X0, P.X1, P.Y0, P.Y1, t0, i, j);
        x[(j - P.Y0) * g.wd + (i - P.X0)] = 1.0;
    }
    if (threadIdx.x == 0) A.passes[gcol] = 0;
}

// ------------------------------------------------------------------ residual
// r = b - A x = -(A x) (x carries the ring data) in FP64, the scaled residual g = S r in
// FP32 for the next solve, |r|^2 per column in a fixed order: a warp per column, lanes
// along the row, rows ascending.  first: |b| = |r| of the initial iterate.  A column stays
// active while |r| > tol |b|.  A CTA takes 8 warps' columns of a chunk, 32 of them or 8
// (blockIdx.y) when the chunks alone would leave SMs idle.
// Bound: the FP64 pipe (busy 82% of the time at 2049^2).  A difference across a face is formed once: the one to the left
// is the left lane's to the right, negated, and the one below is the row below's upward,
// kept in a register; with them a node costs 8 FP64 operations in place of 10.  At 1023^2
// with 169 uneven patches all passes take 27.3 ms, 34.7 with every difference by itself.
__device__ __forceinline__ void residual_done(const DirArgs& A, int gc, double t, int first) {
    const double b2 = first ? t : A.b2[gc];
    if (first) A.b2[gc] = t;
    else A.passes[gc] += 1;
    A.r2[gc] = t;
    A.active[gc] = (b2 > 0.0 && t > A.tol * A.tol * b2) ? 1 : 0;
}

// The initial iterate: zero inside, so only nodes next to the ring have a nonzero
// residual; the others are written as the zeros they are.
__global__ void __launch_bounds__(kDirThreads) direct_residual_first_kernel(DirArgs A, int per) {
    const int4 ch = A.chunks[blockIdx.x];
    const int m = ch.x, c0 = ch.y, nc = ch.z, chunk = ch.w;
    const PatchDev P = A.patches[m];
    const Geo g = geo(P);
    const int n = g.nx, N = A.N;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const double* sv = A.s + A.s_off[m];
    float* Rc = A.R + A.r_off[m] + (long long)chunk * g.ny * kCB * n;
    for (int q = 0; q < per; ++q) {
        const int c = warp + 8 * (per * blockIdx.y + q);
        if (c >= nc) continue;
        const double* x0 = A.X + A.x_off[m] + (long long)(c0 + c) * g.hd * g.wd + g.wd + 1;
        auto residual = [&](int j, int k) {
            const double* x = x0 + (long long)j * g.wd;
            const long long gj = P.Y0 + 1 + j, gi = P.X0 + 1 + k;
            const double ae = A.aE[gj * N + gi], aw = A.aE[gj * N + gi - 1];
            const double an = A.aN[gj * (N + 1) + gi], as = A.aN[(gj - 1) * (N + 1) + gi];
            const double xc = x[k];
            const double r = ae * (x[k + 1] - xc) + aw * (x[k - 1] - xc) + an * (x[k + g.wd] - xc) +
                             as * (x[k - g.wd] - xc);
            Rc[((long long)j * kCB + c) * n + k] = (float)(r * sv[j * n + k]);
            return r;
        };
        double acc = 0.0;
        auto full_row = [&](int j) {
            for (int k = lane; k < n; k += 32) {
                const double r = residual(j, k);
                acc += r * r;
            }
        };
        if (g.ny > 0) full_row(0);
        // rows between: the lanes take 32 rows' first and last nodes at once; the squares are
        // then added row by row in the lanes that hold those nodes
        const int lr = (n - 1) & 31;
        for (int j0 = 1; j0 + 1 < g.ny && n > 0; j0 += 32) {
            const int jn = min(32, g.ny - 1 - j0);
            const double rl = lane < jn ? residual(j0 + lane, 0) : 0.0;
            const double rr = n > 1 && lane < jn ? residual(j0 + lane, n - 1) : 0.0;
            for (int j = 0; j < jn; ++j) {
                const double a = __shfl_sync(0xffffffffu, rl, j), b = __shfl_sync(0xffffffffu, rr, j);
                if (lane == 0) acc += a * a;
                if (n > 1 && lane == lr) acc += b * b;
                float* row = Rc + ((long long)(j0 + j) * kCB + c) * n;
                for (int k = lane; k < n; k += 32)
                    if (k > 0 && k + 1 < n) row[k] = 0.f;
            }
        }
        if (g.ny > 1) full_row(g.ny - 1);
        const double t = warp_sum(acc);
        if (lane == 0) residual_done(A, A.col_base[m] + c0 + c, t, 1);
    }
}

template <int G>
__global__ void __launch_bounds__(kDirThreads) direct_residual_kernel(DirArgs A, int per) {
    const int4 ch = A.chunks[blockIdx.x];
    const int m = ch.x, c0 = ch.y, nc = ch.z, chunk = ch.w;
    const int gbase = A.col_base[m] + c0;
    const PatchDev P = A.patches[m];
    const Geo g = geo(P);
    const int n = g.nx, N = A.N, wd = g.wd;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const double* sv = A.s + A.s_off[m];
    float* Rc = A.R + A.r_off[m] + (long long)chunk * g.ny * kCB * n;
    const double* aEp = A.aE + (long long)(P.Y0 + 1) * N + P.X0 + 1;        // east face of node (0, 0)
    const double* aNp = A.aN + (long long)(P.Y0 + 1) * (N + 1) + P.X0 + 1;  // north face
    for (int q = 0; q < per; ++q) {
        const int c = warp + 8 * (per * blockIdx.y + q);
        if (c >= nc || !A.active[gbase + c]) continue;                      // warp-uniform
        const double* x = A.X + A.x_off[m] + (long long)(c0 + c) * g.hd * wd + wd + 1;   // row 0
        double xc[G], ds[G], an[G];                     // row j; difference and face below it
#pragma unroll
        for (int u = 0; u < G; ++u) {
            const int k = lane + 32 * u;
            xc[u] = k < n ? x[k] : 0.0;
            ds[u] = k < n ? x[k - wd] - xc[u] : 0.0;
            an[u] = k < n ? aNp[k - (N + 1)] : 0.0;
        }
        double acc = 0.0;
        for (int j = 0; j < g.ny; ++j) {
            const double* xr = x + (long long)j * wd;
            const double* ae_r = aEp + (long long)j * N;
            const double* an_r = aNp + (long long)j * (N + 1);
            float* rr = Rc + ((long long)j * kCB + c) * n;
            double left = 0.0;                          // the last difference of the block of 32 before
#pragma unroll
            for (int u = 0; u < G; ++u) {
                const int k = lane + 32 * u;
                const bool in = k < n;
                if (32 * u < n) {
                    const double xe = in ? xr[k + 1] : 0.0, xn = in ? xr[k + wd] : 0.0;
                    const double ae = in ? ae_r[k] : 0.0, aw = in ? ae_r[k - 1] : 0.0;
                    const double anew = in ? an_r[k] : 0.0, s = in ? sv[j * n + k] : 0.0;
                    const double de = xe - xc[u], dn = xn - xc[u];
                    double dw = -__shfl_up_sync(0xffffffffu, de, 1);
                    if (u == 0) {
                        const double w0 = xr[-1] - xc[0];
                        if (lane == 0) dw = w0;
                    } else if (lane == 0) {
                        dw = -left;
                    }
                    left = __shfl_sync(0xffffffffu, de, 31);
                    if (in) {
                        const double r = ae * de + aw * dw + anew * dn + an[u] * ds[u];
                        acc += r * r;
                        rr[k] = (float)(r * s);
                    }
                    ds[u] = -dn;
                    an[u] = anew;
                    xc[u] = xn;
                }
            }
        }
        const double t = warp_sum(acc);
        if (lane == 0) residual_done(A, gbase + c, t, 0);
    }
}

// ------------------------------------------------------------------ solve
// d = Z^{-1} g by the two sweeps for the columns of one CTA, then x += S d.  8 CPW columns
// (two chunks of 32, or one): warp w owns columns CPW w .., lane l the rows l + 32 q, so a
// thread keeps its w_j or d_{j+1} in registers and writes the next product's input y
// straight from them.  W_j streams through a ring of slabs of 32 terms (cp.async, three
// ahead, one barrier per slab); the product reads it four terms at a time (16-byte loads,
// conflict-free) against broadcast loads of y, 4 G CPW FMAs for G + CPW loads, each output
// one chain of FMAs over the terms in order.  R of the next row (forward) or w_j (backward)
// is read before the product that hides it.  Bound: issue slots and the latency of the row
// chain (2 nx^2 FMA per row and column): with 32 columns per CTA on 64 patches 54% of the issue
// slots and 38% of the FP32 pipe are busy, shared and global loads the first stalls; a warp
// whose columns have all converged skips its products.  143356 columns on 1024 patches
// (2049^2): 64 ms for all passes, 17 TFLOP/s, 24% of the FP32 rate; with W_j by plain loads and
// 32 columns per CTA 93 ms.
constexpr int kSlabRows = 32;
constexpr int kSlabs = 4;

__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// floats of shared memory: the slabs (and slack for the padded rows' reads), y
__host__ __device__ inline int solve_smem_floats(int ld, int cw) {
    return kSlabs * kSlabRows * ld + 128 + (ld + 3) / 4 * 4 * cw;
}

template <int G, int CPW>
__global__ void __launch_bounds__(kDirThreads, 2) direct_solve_kernel(DirArgs A) {
    extern __shared__ __align__(16) float ssm[];
    constexpr int CW = 8 * CPW;                         // columns of the CTA
    const int4 ch = A.ctas[blockIdx.x];                 // patch, first column, columns, first chunk
    const int m = ch.x, c0 = ch.y, nc = ch.z, chunk = ch.w;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int* active = A.active + A.col_base[m] + c0;
    unsigned act = 0;                                   // the warp's active columns
#pragma unroll
    for (int c = 0; c < CPW; ++c)
        if (CPW * warp + c < nc && active[CPW * warp + c]) act |= 1u << c;
    if (!__syncthreads_or((int)act)) return;
    const PatchDev P = A.patches[m];
    const Geo g = geo(P);
    const int n = g.nx, ld = g.ld, ny = g.ny;
    if (n < 1 || ny < 1) return;
    float* Ws = ssm;
    float* Ys = Ws + kSlabs * kSlabRows * ld + 128;     // [k][CW], 16-byte groups xor-ed with k mod 8
    const float* Wg = A.W + A.w_off[m];
    const float* Dg = A.D + A.s_off[m];
    const double* sv = A.s + A.s_off[m];
    const float* Rc = A.R + A.r_off[m] + (long long)chunk * ny * kCB * n;
    const long long r_chunk = (long long)ny * kCB * n;
    const int kw = nc > kCB ? 2 * kCB : kCB;            // columns the CTA's part of K holds per row
    float* Kc = A.K + A.k_off[m] + (long long)chunk * ny * ld * kCB;
    const int nks = (n + kSlabRows - 1) / kSlabRows, total = (2 * ny - 1) * nks;
    auto row_of = [&](int t) { return t < ny ? t : 2 * ny - 2 - t; };
    auto issue = [&](int f) {                           // slab f of the stream over both sweeps
        if (f < total) {
            const int t = f / nks, ks = f - t * nks;
            const float* src = Wg + (long long)row_of(t) * ld * ld + ks * kSlabRows * ld;
            float* dst = Ws + (f % kSlabs) * kSlabRows * ld;
            const int count = min(kSlabRows, ld - ks * kSlabRows) * ld;
            for (int e = threadIdx.x * 4; e < count; e += kDirThreads * 4) cp_async16(dst + e, src + e);
        }
        cp_async_commit();
    };
    auto put_y = [&](int i, const float (&v)[CPW]) {
        float* y = Ys + i * CW;
#pragma unroll
        for (int c = 0; c < CPW; c += 4)
            *reinterpret_cast<float4*>(y + ((((CPW * warp + c) >> 2) ^ (i & 7)) << 2)) =
                make_float4(v[c], v[c + 1], v[c + 2], v[c + 3]);
    };
    // R of row j or w of row j for this thread's rows and columns
    float pre[G][CPW];
    auto load_r = [&](int j) {
#pragma unroll
        for (int q = 0; q < G; ++q) {
            const int i = lane + 32 * q;
#pragma unroll
            for (int c = 0; c < CPW; ++c) {
                const int col = CPW * warp + c;
                pre[q][c] = (i < n && (act >> c & 1u))
                                ? Rc[(col / kCB) * r_chunk + ((long long)j * kCB + col % kCB) * n + i] : 0.f;
            }
        }
    };
    for (int f = 0; f < kSlabs - 1; ++f) issue(f);
    load_r(0);
#pragma unroll
    for (int q = 0; q < G; ++q) {
        const int i = lane + 32 * q;
        if (i < (ld + 3) / 4 * 4) {                     // rows n .. of y stay zero
            float v[CPW];
#pragma unroll
            for (int c = 0; c < CPW; ++c) v[c] = i < n ? pre[q][c] : 0.f;
            put_y(i, v);
        }
    }
    int f = 0;
    for (int t = 0; t < 2 * ny - 1; ++t) {
        const int j = row_of(t);
        const bool fwd = t < ny, turn = t == ny - 1;
        if (fwd) {
            if (!turn) load_r(j + 1);
        } else {
            // the iterate's row into the L2: two 128-byte lines per 32 values
#pragma unroll
            for (int c = 0; c < CPW; ++c)
                if (act >> c & 1u) {
                    const double* xr = A.X + A.x_off[m] + (long long)(c0 + CPW * warp + c) * g.hd * g.wd + (j + 1) * g.wd + 1;
                    if (16 * lane < n) asm volatile("prefetch.global.L2 [%0];" ::"l"(xr + 16 * lane));
                }
#pragma unroll
            for (int q = 0; q < G; ++q) {
                const int i = lane + 32 * q;
#pragma unroll
                for (int c = 0; c < CPW; ++c)
                    pre[q][c] = (i < n && (act >> c & 1u)) ? Kc[((long long)j * kw + CPW * warp + c) * ld + i] : 0.f;
            }
        }
        float acc[G][CPW];
#pragma unroll
        for (int q = 0; q < G; ++q)
#pragma unroll
            for (int c = 0; c < CPW; ++c) acc[q][c] = 0.f;
        for (int ks = 0; ks < nks; ++ks, ++f) {
            cp_async_wait<kSlabs - 2>();
            __syncthreads();                            // slab f (and y) visible, slab f - 1 no longer read
            issue(f + kSlabs - 1);
            if (!act) continue;
            const float* Wk = Ws + (f % kSlabs) * kSlabRows * ld;
            const int kn4 = min(kSlabRows, ld - ks * kSlabRows) / 4;
            for (int k4 = 0; k4 < kn4; ++k4) {
                float4 w[G];
#pragma unroll
                for (int q = 0; q < G; ++q) w[q] = *reinterpret_cast<const float4*>(Wk + (k4 * ld + lane + 32 * q) * 4);
#pragma unroll
                for (int kk = 0; kk < 4; ++kk) {
                    const int k = ks * kSlabRows + 4 * k4 + kk;
                    float y[CPW];
#pragma unroll
                    for (int c = 0; c < CPW; c += 4) {
                        const float4 v = *reinterpret_cast<const float4*>(
                            Ys + k * CW + ((((CPW * warp + c) >> 2) ^ (k & 7)) << 2));
                        y[c] = v.x; y[c + 1] = v.y; y[c + 2] = v.z; y[c + 3] = v.w;
                    }
#pragma unroll
                    for (int q = 0; q < G; ++q) {
                        const float wv = kk == 0 ? w[q].x : kk == 1 ? w[q].y : kk == 2 ? w[q].z : w[q].w;
#pragma unroll
                        for (int c = 0; c < CPW; ++c) acc[q][c] = fmaf(wv, y[c], acc[q][c]);
                    }
                }
            }
        }
        __syncthreads();                                // y no longer read
        // forward: w_j = acc; backward: d_j = acc + w_j (at the turn 0 + w_j)
#pragma unroll
        for (int q = 0; q < G; ++q) {
            const int i = lane + 32 * q;
            if (i >= n || !act) continue;
            const bool next = fwd ? true : j > 0;
            float dn = 0.f;                             // coupling of the next product's row
            if (fwd && !turn) dn = Dg[j * n + i];
            else if (j > 0) dn = Dg[(j - 1) * n + i];
            float v[CPW];
            if (fwd && !turn) {
#pragma unroll
                for (int c = 0; c < CPW; ++c) {
                    const float w = acc[q][c];
                    if (act >> c & 1u) Kc[((long long)j * kw + CPW * warp + c) * ld + i] = w;
                    v[c] = (act >> c & 1u) ? fmaf(dn, w, pre[q][c]) : 0.f;
                }
            } else {
                const double s = sv[j * n + i];
#pragma unroll
                for (int c = 0; c < CPW; ++c) {
                    const float dv = turn ? 0.f + acc[q][c] : acc[q][c] + pre[q][c];
                    if (act >> c & 1u) {
                        double* x = A.X + A.x_off[m] + (long long)(c0 + CPW * warp + c) * g.hd * g.wd + (j + 1) * g.wd + 1 + i;
                        *x += s * (double)dv;
                    }
                    v[c] = (act >> c & 1u) ? dn * dv : 0.f;
                }
            }
            if (next) put_y(i, v);
        }
    }
    cp_async_wait<0>();
}

// ------------------------------------------------------------------ finish
// One CTA per column: restriction to K_m and the column's statistics.
__global__ void __launch_bounds__(kDirThreads) direct_finish_kernel(DirArgs A) {
    const int gcol = A.col0 + blockIdx.x;
    const int2 mc = A.cols[gcol];
    const int m = mc.x, col = mc.y;
    const PatchDev P = A.patches[m];
    const Geo g = geo(P);
    const double* x = A.X + A.x_off[m] + (long long)col * g.hd * g.wd;
    const int wk = P.x1 - P.x0 + 1;
    double* out = A.snaps + P.snap_offset + (long long)col * P.n_k;
    for (int t = threadIdx.x; t < P.n_k; t += blockDim.x) {
        const int jj = t / wk, ii = t - jj * wk;
        out[t] = x[(P.y0 - P.Y0 + jj) * g.wd + (P.x0 - P.X0 + ii)];
    }
    if (threadIdx.x == 0) {
        const int si = A.stat_idx[gcol];
        const int ps = A.passes[gcol];
        A.stats[3 * si + 0] = ps;
        A.stats[3 * si + 1] = ps;
        A.stats[3 * si + 2] = A.active[gcol] ? 1 : 0;
    }
}

// Tables and buffers of the direct solver (once per medium).
msp_status direct_plan(Medium& M, cudaStream_t s) {
    Medium::Direct& D = M.dir;
    if (D.planned) return MSP_OK;
    const int np = (int)M.patches.size();
    std::vector<long long> w_off(np), s_off(np), x_off(np), r_off(np), k_off(np);
    std::vector<int> col_base(np);
    std::vector<int2> cols;
    std::vector<int4> chunks;
    long long w = 0, sv = 0, x = 0, r = 0, k = 0;
    int max_ld = 0;
    for (int m = 0; m < np; ++m) {
        const PatchDev& P = M.patches[m];
        const Geo g = geo(P);
        const int nch = (P.cols + kCB - 1) / kCB;
        w_off[m] = w; s_off[m] = sv; x_off[m] = x; r_off[m] = r; k_off[m] = k;
        col_base[m] = (int)cols.size();
        const long long nx = std::max(g.nx, 0), ny = std::max(g.ny, 0);
        w += ny * g.ld * g.ld;
        sv += ny * nx;
        x += (long long)P.cols * g.hd * g.wd;
        r += (long long)nch * ny * kCB * nx;
        k += (long long)nch * ny * g.ld * kCB;
        for (int c = 0; c < P.cols; ++c) cols.push_back(make_int2(m, c));
        for (int q = 0; q < nch; ++q) chunks.push_back(make_int4(m, q * kCB, std::min(kCB, P.cols - q * kCB), q));
        max_ld = std::max(max_ld, g.ld);
    }
    // statistics slot of every column: its position in the mixed-precision item order
    std::vector<int> stat_idx(cols.size(), 0);
    const std::vector<int2>& order = M.items_prec_host[1];
    for (size_t i = 0; i < order.size(); ++i) stat_idx[col_base[order[i].x] + order[i].y] = (int)i;
    D.n_cols = (int)cols.size();
    D.n_chunks = (int)chunks.size();
    D.max_nxp = max_ld;
    // CTAs of the sweeps: pairs of chunks (64 columns) where those fill the GPU twice, single
    // chunks otherwise (a small medium then spreads over more SMs)
    std::vector<int4> ctas;
    for (size_t q = 0; q < chunks.size(); ++q) {
        const bool two = q + 1 < chunks.size() && chunks[q + 1].x == chunks[q].x;
        ctas.push_back(make_int4(chunks[q].x, chunks[q].y, chunks[q].z + (two ? chunks[q + 1].z : 0), chunks[q].w));
        if (two) ++q;
    }
    D.wide = (int)ctas.size() >= 2 * num_sms();
    if (!D.wide) ctas = chunks;
    D.n_ctas = (int)ctas.size();
    // Two groups of patches with half of the columns each, on two streams: the residuals
    // of one (FP64 pipe) run beside the sweeps of the other (FP32 pipe, load latency).
    // One group where half of the sweeps' CTAs would not fill the GPU twice.
    D.groups.assign(2, Medium::Direct::Group{});
    Medium::Direct::Group& g0 = D.groups[0];
    Medium::Direct::Group& g1 = D.groups[1];
    int half = np;
    if (D.n_ctas >= 4 * num_sms())
        for (half = 0; half < np && 2 * col_base[half] < (int)cols.size(); ++half) {}
    auto below = [half](const std::vector<int4>& v) {
        return (int)(std::find_if(v.begin(), v.end(), [half](const int4& e) { return e.x >= half; }) - v.begin());
    };
    const int hc = below(chunks), ha = below(ctas), hcol = half < np ? col_base[half] : (int)cols.size();
    g0 = {0, half, 0, hcol, 0, hc, 0, ha};
    g1 = {half, np - half, hcol, (int)cols.size() - hcol, hc, (int)chunks.size() - hc, ha, (int)ctas.size() - ha};
    if (g1.patches == 0) {
        D.groups.pop_back();
    } else if (!D.side) {
        MSP_CUDA(cudaStreamCreateWithFlags(&D.side, cudaStreamNonBlocking));
        MSP_CUDA(cudaEventCreateWithFlags(&D.fork, cudaEventDisableTiming));
        MSP_CUDA(cudaEventCreateWithFlags(&D.join, cudaEventDisableTiming));
    }
    const int ts = std::max(1, (max_ld + 15) / 16);
    D.factor_smem_max = (int)sizeof(float) * (max_ld * (max_ld + 1) + 2 * ts * 16 * ts);
    D.chunk_smem_max = (int)sizeof(float) * solve_smem_floats(max_ld, D.wide ? 2 * kCB : kCB);
    D.w_elems = w; D.s_elems = sv; D.x_elems = x; D.r_elems = r; D.k_elems = k;
    MSP_TRY(upload(D.w_off, w_off, s));
    MSP_TRY(upload(D.s_off, s_off, s));
    MSP_TRY(upload(D.x_off, x_off, s));
    MSP_TRY(upload(D.r_off, r_off, s));
    MSP_TRY(upload(D.k_off, k_off, s));
    MSP_TRY(upload(D.col_base, col_base, s));
    MSP_TRY(upload(D.cols, cols, s));
    MSP_TRY(upload(D.chunks, chunks, s));
    MSP_TRY(upload(D.ctas, ctas, s));
    MSP_TRY(upload(D.stat_idx, stat_idx, s));
    MSP_TRY(D.W.alloc(std::max<long long>(1, w), s));
    MSP_TRY(D.s.alloc(std::max<long long>(1, sv), s));
    MSP_TRY(D.D.alloc(std::max<long long>(1, sv), s));
    MSP_TRY(D.X.alloc(std::max<long long>(1, x), s));
    MSP_TRY(D.R.alloc(std::max<long long>(1, r), s));
    MSP_TRY(D.K.alloc(std::max<long long>(1, k), s));
    MSP_TRY(D.b2.alloc(std::max(1, D.n_cols), s));
    MSP_TRY(D.r2.alloc(std::max(1, D.n_cols), s));
    MSP_TRY(D.active.alloc(std::max(1, D.n_cols), s));
    MSP_TRY(D.passes.alloc(std::max(1, D.n_cols), s));
    MSP_CUDA(cudaStreamSynchronize(s));   // the host tables above go out of scope
    D.planned = true;
    return MSP_OK;
}

DirArgs direct_args(Medium& M, const LocalSolveCfg& cfg) {
    Medium::Direct& D = M.dir;
    DirArgs A{};
    A.N = M.N;
    A.aE = M.aE.p;
    A.aN = M.aN.p;
    A.patches = M.patches_dev.p;
    A.bpos = M.bpos_dev.p;
    A.seed = cfg.seed;
    A.w_off = D.w_off.p; A.s_off = D.s_off.p; A.x_off = D.x_off.p; A.r_off = D.r_off.p; A.k_off = D.k_off.p;
    A.col_base = D.col_base.p;
    A.cols = D.cols.p;
    A.chunks = D.chunks.p;
    A.ctas = D.ctas.p;
    A.stat_idx = D.stat_idx.p;
    A.W = D.W.p; A.D = D.D.p; A.R = D.R.p; A.K = D.K.p;
    A.s = D.s.p; A.X = D.X.p; A.b2 = D.b2.p; A.r2 = D.r2.p;
    A.active = D.active.p; A.passes = D.passes.p;
    A.snaps = M.snaps.p;
    A.stats = M.item_stats.p;
    A.tol = cfg.tol;
    return A;
}

// phases of the optional timing
enum { kPhFactor = 0, kPhInit = 1, kPhResidual = 2, kPhSolve = 3, kPhFinish = 4, kPhases = 5 };

// start (begin = true) or stop an event pair of phase ph
msp_status mark(Medium::Direct& D, int ph, bool begin, cudaStream_t s) {
    if (!D.timing) return MSP_OK;
    if (begin) {
        while ((int)D.ev.size() < D.ev_used + 2) {
            cudaEvent_t e;
            MSP_CUDA(cudaEventCreate(&e));
            D.ev.push_back(e);
            D.ev_phase.push_back(0);
        }
        D.ev_phase[D.ev_used] = ph;
        MSP_CUDA(cudaEventRecord(D.ev[D.ev_used], s));
    } else {
        MSP_CUDA(cudaEventRecord(D.ev[D.ev_used + 1], s));
        D.ev_used += 2;
    }
    return MSP_OK;
}

template <int G, int CPW>
msp_status launch_solve_g(const DirArgs& A, int grid, int smem, cudaStream_t s) {
    MSP_TRY(allow_smem(direct_solve_kernel<G, CPW>, smem));
    direct_solve_kernel<G, CPW><<<grid, kDirThreads, smem, s>>>(A);
    count_launches(1);
    return MSP_OK;
}

template <int CPW>
msp_status launch_solve(const DirArgs& A, int G, int grid, int smem, cudaStream_t s) {
    switch (G) {
        case 1: return launch_solve_g<1, CPW>(A, grid, smem, s);
        case 2: return launch_solve_g<2, CPW>(A, grid, smem, s);
        case 3: return launch_solve_g<3, CPW>(A, grid, smem, s);
        case 4: return launch_solve_g<4, CPW>(A, grid, smem, s);
        default: return launch_solve_g<5, CPW>(A, grid, smem, s);
    }
}

}  // namespace

bool direct_fits(const Medium& M) {
    for (const PatchDev& P : M.patches) {
        const Geo g = geo(P);
        if (g.ld > kDirMaxLd) return false;
    }
    return !M.patches.empty();
}

template <int TS>
static msp_status launch_factor(const DirArgs& A, int np, int smem, cudaStream_t s) {
    MSP_TRY(allow_smem(direct_factor_kernel<TS>, smem));
    direct_factor_kernel<TS><<<np, kDirThreads, smem, s>>>(A);
    return MSP_OK;
}

// Factor (once per medium), residuals, sweeps and restriction of one group of patches.
static msp_status launch_group(Medium::Direct& D, const Medium::Direct::Group& grp, DirArgs A, const LocalSolveCfg& cfg,
                               cudaStream_t s) {
    A.patch0 = grp.patch0;
    A.col0 = grp.col0;
    A.chunks += grp.chunk0;
    A.ctas += grp.cta0;
    if (!D.factored) {
        MSP_TRY(mark(D, kPhFactor, true, s));
        // one sub-block size for the launch, from the widest padded row
        switch (std::max(1, (D.max_nxp + 15) / 16)) {
            case 1: MSP_TRY(launch_factor<1>(A, grp.patches, D.factor_smem_max, s)); break;
            case 2: MSP_TRY(launch_factor<2>(A, grp.patches, D.factor_smem_max, s)); break;
            case 3: MSP_TRY(launch_factor<3>(A, grp.patches, D.factor_smem_max, s)); break;
            case 4: MSP_TRY(launch_factor<4>(A, grp.patches, D.factor_smem_max, s)); break;
            case 5: MSP_TRY(launch_factor<5>(A, grp.patches, D.factor_smem_max, s)); break;
            case 6: MSP_TRY(launch_factor<6>(A, grp.patches, D.factor_smem_max, s)); break;
            case 7: MSP_TRY(launch_factor<7>(A, grp.patches, D.factor_smem_max, s)); break;
            case 8: MSP_TRY(launch_factor<8>(A, grp.patches, D.factor_smem_max, s)); break;
            case 9: MSP_TRY(launch_factor<9>(A, grp.patches, D.factor_smem_max, s)); break;
            default: MSP_TRY(launch_factor<10>(A, grp.patches, D.factor_smem_max, s)); break;
        }
        count_launches(1);
        MSP_TRY(mark(D, kPhFactor, false, s));
        MSP_CUDA(cudaGetLastError());
    }
    if (grp.cols == 0) return MSP_OK;
    MSP_TRY(mark(D, kPhInit, true, s));
    direct_init_kernel<<<grp.cols, kDirThreads, 0, s>>>(A);
    count_launches(1);
    MSP_TRY(mark(D, kPhInit, false, s));
    MSP_TRY(mark(D, kPhResidual, true, s));
    // columns per warp of the residual: 4 (a chunk per CTA), or 1 while that fills the GPU less
    // than six CTAs per SM
    const int per = grp.chunks >= 6 * num_sms() ? 4 : 1;
    const dim3 rgrid(grp.chunks, 4 / per);
    direct_residual_first_kernel<<<rgrid, kDirThreads, 0, s>>>(A, per);
    count_launches(1);
    MSP_TRY(mark(D, kPhResidual, false, s));
    MSP_CUDA(cudaGetLastError());
    const int G = std::max(1, (D.max_nxp + 31) / 32);
    const int passes = std::max(1, std::min(cfg.max_ref, kDirMaxPasses));
    for (int p = 0; p < passes; ++p) {
        MSP_TRY(mark(D, kPhSolve, true, s));
        if (D.wide) MSP_TRY(launch_solve<8>(A, G, grp.ctas, D.chunk_smem_max, s));
        else MSP_TRY(launch_solve<4>(A, G, grp.ctas, D.chunk_smem_max, s));
        MSP_TRY(mark(D, kPhSolve, false, s));
        MSP_TRY(mark(D, kPhResidual, true, s));
        switch (G) {
            case 1: direct_residual_kernel<1><<<rgrid, kDirThreads, 0, s>>>(A, per); break;
            case 2: direct_residual_kernel<2><<<rgrid, kDirThreads, 0, s>>>(A, per); break;
            case 3: direct_residual_kernel<3><<<rgrid, kDirThreads, 0, s>>>(A, per); break;
            case 4: direct_residual_kernel<4><<<rgrid, kDirThreads, 0, s>>>(A, per); break;
            default: direct_residual_kernel<5><<<rgrid, kDirThreads, 0, s>>>(A, per); break;
        }
        count_launches(1);
        MSP_TRY(mark(D, kPhResidual, false, s));
        MSP_CUDA(cudaGetLastError());
    }
    MSP_TRY(mark(D, kPhFinish, true, s));
    direct_finish_kernel<<<grp.cols, kDirThreads, 0, s>>>(A);
    count_launches(1);
    MSP_TRY(mark(D, kPhFinish, false, s));
    MSP_CUDA(cudaGetLastError());
    return MSP_OK;
}

msp_status launch_local_solves_direct(Medium& M, const LocalSolveCfg& cfg, cudaStream_t s) {
    if (!direct_fits(M)) {
        set_error("direct local solver: a buffered patch is wider than 160 interior nodes");
        return MSP_ERR_INVALID_ARG;
    }
    MSP_TRY(direct_plan(M, s));
    Medium::Direct& D = M.dir;
    const DirArgs A0 = direct_args(M, cfg);
    D.ev_used = 0;
    // phase timing reads one stream's events: the groups then run one after the other
    const bool forked = D.groups.size() > 1 && !D.timing;
    if (forked) {
        MSP_CUDA(cudaEventRecord(D.fork, s));
        MSP_CUDA(cudaStreamWaitEvent(D.side, D.fork, 0));
    }
    msp_status st = MSP_OK;
    for (size_t q = 0; q < D.groups.size() && st == MSP_OK; ++q)
        st = launch_group(D, D.groups[q], A0, cfg, forked && q > 0 ? D.side : s);
    if (forked) {   // also after an error: the caller's stream waits for what was launched
        MSP_CUDA(cudaEventRecord(D.join, D.side));
        MSP_CUDA(cudaStreamWaitEvent(s, D.join, 0));
    }
    MSP_TRY(st);
    D.factored = true;
    MSP_CUDA(cudaGetLastError());
    return MSP_OK;
}

}  // namespace msp

using namespace msp;

extern "C" msp_status msp_medium_set_timing(msp_medium m, int enable) {
    clear_error();
    MSP_CHECK_ARG(m, "msp_medium_set_timing: NULL medium");
    m->M.dir.timing = enable != 0;
    m->M.dir.ev_used = 0;
    return MSP_OK;
}

extern "C" msp_status msp_medium_direct_timing(msp_medium m, double* ms_host, int* launches_host) {
    clear_error();
    MSP_CHECK_ARG(m && ms_host, "msp_medium_direct_timing: NULL argument");
    Medium::Direct& D = m->M.dir;
    for (int p = 0; p < kPhases; ++p) {
        ms_host[p] = 0.0;
        if (launches_host) launches_host[p] = 0;
    }
    for (int i = 0; i + 1 < D.ev_used; i += 2) {
        MSP_CUDA(cudaEventSynchronize(D.ev[i + 1]));
        float t = 0.f;
        MSP_CUDA(cudaEventElapsedTime(&t, D.ev[i], D.ev[i + 1]));
        ms_host[D.ev_phase[i]] += t;
        if (launches_host) launches_host[D.ev_phase[i]] += 1;
    }
    return MSP_OK;
}
