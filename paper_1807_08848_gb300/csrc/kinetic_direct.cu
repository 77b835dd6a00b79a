// Direct local solver of the kinetic slab (Sec. 4, Eq. RTE with the
// Henyey-Greenstein collision of Eq. HG; the offline local problem of
// Eq. rte_random on a buffered patch).
//
// Discrete operator on the nodes i = 0..nn-1 of a buffered patch, unknowns
// f_i in R^{n_v} at every node (the incoming components at the two ends carry
// identity rows whose right-hand side is the random datum):
//
//   D_i f_i + L_i f_{i-1} + U_i f_{i+1} = b_i,
//   D_i = diag(a_l + sigma_l/eps) - Kw/eps,    a_l = |v_l|/dx,
//   L_i = -diag(a_l [v_l > 0]),  U_i = -diag(a_l [v_l < 0]).
//
// Block LU over the nodes: S_0 = D_0, S_i = D_i - L_i S_{i-1}^{-1} U_{i-1}; the
// coupling touches only the (v>0 rows, v<0 columns) quadrant.  Every S_i is a
// nonsingular M-matrix (weakly row-diagonally dominant since the gain row sums
// equal the loss rates, strictly at the identity rows), so neither the block
// elimination nor the Gauss-Jordan inversion of each S_i needs pivoting.  The
// factor keeps W_i = S_i^{-1} for every node, formed in halves of the velocities.
//
// The solve kernel takes one CTA per (patch, 16 samples), one sample per lane,
// and refines in FP64: r = b - A f (FP64, sweeping a three-node window of f
// through shared memory), forward y_i = W_i (r_i - L_i y_{i-1}), backward
// x_i = y_i - W_i U_i x_{i+1}, f += x.  With the FP64 factor one pass solves
// and a second confirms; with the FP32 factor each pass gains about seven
// digits.  Stop when max |r_l| / D_ll <= tol max |f|.
#include "kinetic_internal.h"
#include "device_util.cuh"

#include <algorithm>
#include <cmath>

namespace msp {
namespace {

constexpr int kKdThreads = 256;
constexpr int kKdG = 16;        // samples per CTA of the solve, one per lane of a half-warp
constexpr int kKdHalves = kKdThreads / kKdG;   // half-warps of a CTA
constexpr int kKdLd = 17;       // padded row stride of the [velocity][sample] tiles
constexpr int kKdMaxNv = 128;
constexpr int kKdMaxPasses = 16;   // corrections per solve at most

struct KdArgs {
    int N, n_v, S, max_passes;
    double eps, tol;
    uint64_t seed;
    const double* v;
    const double* Kw;
    const double* sigma;
    const KPatchDev* patches;
    const long long* node_off;
    double* f;
    double* snaps;
    int* stats;
};

__device__ __forceinline__ bool kd_identity(int i, int nn, double vl) {
    return (i == 0 && vl > 0.0) || (i == nn - 1 && vl < 0.0);
}

// The factor in halves.  With the h = n_v/2 negative velocities first, S_i = [A B; C D],
// and of the interior nodes' blocks only C depends on the node:
//
//   C_i = C_0 - a_+ (W_{i-1})_{+-} a_-,   X_i = D^{-1} C_i = X_0 + F P_{i-1} a_-,
//   E_i = A - B X_i,   P_i = X_i E_i^{-1},   F = D^{-1} a_+,   G = B D^{-1},
//   W_i = [ E^{-1}, -E^{-1} G ; -P, D^{-1} + P G ]
//
// (end nodes: C = 0, D = I at the first, A = I, B = 0 at the last).  E is a Schur
// complement of an M-matrix, so it needs no pivoting either.  A node's serial part is one
// h x h inverse and three h x h products instead of an n_v x n_v inverse, 4 h^3 for 8 h^3
// multiply-adds and h barriers for 2 h; the + columns of W, 2 h^3, are independent of each
// other over all nodes and run on the whole GPU.
struct KdHalf {   // offsets (in h*h) of the node-independent blocks
    static constexpr int kA = 0, kB = 1, kDinv = 2, kG = 3, kX0 = 4, kF = 5, kCount = 6;
};
constexpr int kKdMaxHalf = kKdMaxNv / 2;

// The blocks that no node changes, by one CTA: D inverted by Gauss-Jordan in shared memory
// (one thread takes each pivot's reciprocal), then G, X_0 and F.
template <class T>
__global__ void __launch_bounds__(1024) kd_blocks_kernel(KdArgs A, T* __restrict__ out) {
    extern __shared__ __align__(16) unsigned char kd_dyn[];
    double* D = reinterpret_cast<double*>(kd_dyn);   // h x h
    __shared__ double col[kKdMaxHalf], row[kKdMaxHalf], rcp;
    const int nv = A.n_v, h = nv / 2, hh = h * h;
    const double dx = 1.0 / A.N, ie = 1.0 / A.eps;
    auto entry = [&](int r, int c) {   // interior row r, without the neighbours' term
        double s = -ie * A.Kw[(long long)r * nv + c];
        if (r == c) s += fabs(A.v[r]) / dx + ie * A.sigma[r];
        return s;
    };
    for (int e = threadIdx.x; e < hh; e += blockDim.x) {
        const int r = e / h, c = e % h;
        D[e] = entry(h + r, h + c);
        out[KdHalf::kA * hh + e] = (T)entry(r, c);
        out[KdHalf::kB * hh + e] = (T)entry(r, h + c);
    }
    __syncthreads();
    for (int k = 0; k < h; ++k) {
        if (threadIdx.x < h) {
            col[threadIdx.x] = D[threadIdx.x * h + k];
            row[threadIdx.x] = D[k * h + threadIdx.x];
        }
        if (threadIdx.x == 0) rcp = 1.0 / D[k * h + k];
        __syncthreads();
        for (int e = threadIdx.x; e < hh; e += blockDim.x) {
            const int r = e / h, c = e % h;
            const double cr = col[r] * rcp;
            double x = D[e];
            if (r != k) x = (c != k) ? fma(-cr, row[c], x) : -cr;
            else x = (c != k) ? row[c] * rcp : rcp;
            D[e] = x;
        }
        __syncthreads();
    }
    for (int e = threadIdx.x; e < hh; e += blockDim.x) {
        const int r = e / h, c = e % h;
        double g = 0.0, x = 0.0;
        for (int k = 0; k < h; ++k) {
            g = fma(entry(r, h + k), D[k * h + c], g);
            x = fma(D[r * h + k], entry(h + k, c), x);
        }
        out[KdHalf::kDinv * hh + e] = (T)D[e];
        out[KdHalf::kG * hh + e] = (T)g;
        out[KdHalf::kX0 * hh + e] = (T)x;
        out[KdHalf::kF * hh + e] = (T)(D[e] * (fabs(A.v[h + c]) / dx));
    }
}

// acc[a][b] += sum_k L[ty + 16 a][k] R[k][tx + 16 b] of h x h blocks in shared memory with
// row stride ld (entries beyond h are left alone).
template <class T, int RA>
__device__ __forceinline__ void kd_product(T (&acc)[RA][RA], const T* L, const T* R, int h, int ld, int tx, int ty) {
    for (int k = 0; k < h; ++k) {
        T l[RA], r[RA];
#pragma unroll
        for (int a = 0; a < RA; ++a) {
            l[a] = (ty + 16 * a < h) ? L[(ty + 16 * a) * ld + k] : T(0);
            r[a] = (tx + 16 * a < h) ? R[k * ld + tx + 16 * a] : T(0);
        }
#pragma unroll
        for (int a = 0; a < RA; ++a)
#pragma unroll
            for (int b = 0; b < RA; ++b) acc[a][b] += l[a] * r[b];
    }
}

// The serial part, one CTA per patch: E_i, its inverse and P_i of every node, written to the
// - columns of W.  Thread (ty, tx) of the 16 x 16 grid owns the entries (ty + 16 a,
// tx + 16 b), a, b < RA, of each h x h block (h <= 16 RA).  Bound by FP64 issue of the SMs that
// hold a patch (their pipe is busy 74% of the time, 31% over the GPU at 64 patches): a warp's
// instruction holds its quarter of the SM for 64 clocks, a division for about 380, so only
// the thread that finishes the next pivot divides and publishes the reciprocal.  8193
// nodes, 64 velocities, 64 patches: the factor as one n_v x n_v inverse per node took
// 42 ms of a pass of 114.2; with the halves it takes 13.2, the pass 85.4.
template <class T, int RA>
__global__ void __launch_bounds__(kKdThreads) kd_chain_kernel(KdArgs A, const T* __restrict__ blocks, T* W) {
    extern __shared__ __align__(16) unsigned char kd_dyn[];
    __shared__ T colk[2][kKdMaxHalf], rowk[2][kKdMaxHalf], rcp[2];
    const int m = blockIdx.x, nv = A.n_v, h = nv / 2, hh = h * h, ld = h + 1;
    T* sB = reinterpret_cast<T*>(kd_dyn);
    T* sF = sB + h * ld;
    T* sX = sF + h * ld;   // X_i
    T* sE = sX + h * ld;   // E_i^{-1}, then P_i a_-
    const KPatchDev P = A.patches[m];
    const int nn = P.X1 - P.X0 + 1;
    const long long n2 = (long long)nv * nv;
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    T* Wm = W + A.node_off[m] * n2;
    for (int e = threadIdx.x; e < hh; e += kKdThreads) {
        const int q = (e / h) * ld + e % h;
        sB[q] = blocks[KdHalf::kB * hh + e];
        sF[q] = blocks[KdHalf::kF * hh + e];
        sX[q] = T(0);   // C = 0 at the first node
    }
    T a0[RA][RA], x0[RA][RA], am[RA];
#pragma unroll
    for (int a = 0; a < RA; ++a) {
        am[a] = (tx + 16 * a < h) ? (T)(fabs(A.v[tx + 16 * a]) * (double)A.N) : T(0);
#pragma unroll
        for (int b = 0; b < RA; ++b) {
            const bool in = ty + 16 * a < h && tx + 16 * b < h;
            const int e = (ty + 16 * a) * h + tx + 16 * b;
            a0[a][b] = in ? blocks[KdHalf::kA * hh + e] : T(0);
            x0[a][b] = in ? blocks[KdHalf::kX0 * hh + e] : T(0);
        }
    }
    __syncthreads();
    // publishes column k, row k and 1 / pivot of the block in x
    auto publish = [&](const T (&x)[RA][RA], int k, int par) {
        const int kq = k >> 4;
        if (tx == (k & 15)) {
#pragma unroll
            for (int a = 0; a < RA; ++a)
#pragma unroll
                for (int b = 0; b < RA; ++b)
                    if (b == kq && ty + 16 * a < h) colk[par][ty + 16 * a] = x[a][b];
        }
        if (ty == (k & 15)) {
#pragma unroll
            for (int a = 0; a < RA; ++a)
#pragma unroll
                for (int b = 0; b < RA; ++b)
                    if (a == kq && tx + 16 * b < h) {
                        rowk[par][tx + 16 * b] = x[a][b];
                        if (b == kq && tx == (k & 15)) rcp[par] = T(1) / x[a][b];
                    }
        }
    };
    for (int i = 0; i < nn; ++i) {
        T x[RA][RA];
#pragma unroll
        for (int a = 0; a < RA; ++a)
#pragma unroll
            for (int b = 0; b < RA; ++b) x[a][b] = T(0);
        if (i == nn - 1) {
#pragma unroll
            for (int a = 0; a < RA; ++a)
#pragma unroll
                for (int b = 0; b < RA; ++b) x[a][b] = (ty + 16 * a == tx + 16 * b) ? T(1) : T(0);
        } else {
            if (i > 0) kd_product<T, RA>(x, sB, sX, h, ld, tx, ty);
#pragma unroll
            for (int a = 0; a < RA; ++a)
#pragma unroll
                for (int b = 0; b < RA; ++b) x[a][b] = a0[a][b] - x[a][b];
            publish(x, 0, 0);
            for (int k = 0; k < h; ++k) {
                const int par = k & 1;
                __syncthreads();
                const T p = rcp[par];
#pragma unroll
                for (int a = 0; a < RA; ++a) {
                    const int r = ty + 16 * a;
                    if (r >= h) continue;
                    const T cr = colk[par][r] * p;
#pragma unroll
                    for (int b = 0; b < RA; ++b) {
                        const int c = tx + 16 * b;
                        if (c >= h) continue;
                        if (r == k) x[a][b] = (c == k) ? p : rowk[par][c] * p;
                        else x[a][b] = (c == k) ? -cr : x[a][b] - cr * rowk[par][c];
                    }
                }
                if (k + 1 < h) publish(x, k + 1, par ^ 1);
            }
        }
        T* Wi = Wm + (long long)i * n2;
#pragma unroll
        for (int a = 0; a < RA; ++a)
#pragma unroll
            for (int b = 0; b < RA; ++b) {
                const int r = ty + 16 * a, c = tx + 16 * b;
                if (r < h && c < h) {
                    sE[r * ld + c] = x[a][b];
                    Wi[(long long)r * nv + c] = x[a][b];
                }
            }
        __syncthreads();
        T pr[RA][RA];
#pragma unroll
        for (int a = 0; a < RA; ++a)
#pragma unroll
            for (int b = 0; b < RA; ++b) pr[a][b] = T(0);
        if (i > 0) kd_product<T, RA>(pr, sX, sE, h, ld, tx, ty);
        __syncthreads();   // every thread is done with E^{-1} and X_i
#pragma unroll
        for (int a = 0; a < RA; ++a)
#pragma unroll
            for (int b = 0; b < RA; ++b) {
                const int r = ty + 16 * a, c = tx + 16 * b;
                if (r < h && c < h) {
                    Wi[(long long)(h + r) * nv + c] = -pr[a][b];
                    sE[r * ld + c] = pr[a][b] * am[b];
                }
            }
        if (i == nn - 1) break;
        __syncthreads();
        T xn[RA][RA];
#pragma unroll
        for (int a = 0; a < RA; ++a)
#pragma unroll
            for (int b = 0; b < RA; ++b) xn[a][b] = x0[a][b];
        if (i > 0) kd_product<T, RA>(xn, sF, sE, h, ld, tx, ty);
#pragma unroll
        for (int a = 0; a < RA; ++a)
#pragma unroll
            for (int b = 0; b < RA; ++b) {
                const int r = ty + 16 * a, c = tx + 16 * b;
                if (r < h && c < h) sX[r * ld + c] = xn[a][b];
            }
        __syncthreads();
    }
}

// The + columns of W of every node, from its - columns: CTA x of a patch's `per` takes the
// nodes x, x + per, ... of the patch with G in shared memory; the - columns pass through it
// too.  blockIdx.x numbers the CTAs patch by patch: a second grid dimension ends at 65535.
template <class T, int RA>
__global__ void __launch_bounds__(kKdThreads) kd_columns_kernel(KdArgs A, const T* __restrict__ blocks, T* W, int per) {
    extern __shared__ __align__(16) unsigned char kd_dyn[];
    const int m = blockIdx.x / per, nv = A.n_v, h = nv / 2, hh = h * h, ld = h + 1;
    T* sG = reinterpret_cast<T*>(kd_dyn);
    T* sL = sG + h * ld;   // 2 h rows: E^{-1} over -P
    const KPatchDev P = A.patches[m];
    const int nn = P.X1 - P.X0 + 1;
    const long long n2 = (long long)nv * nv;
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    T* Wm = W + A.node_off[m] * n2;
    int held = -1;   // 0: B (the first node, where D = I), 1: G
    for (int i = blockIdx.x - m * per; i < nn; i += per) {
        T* Wi = Wm + (long long)i * n2;
        const int want = i > 0;
        __syncthreads();   // the previous node's products are done
        if (held != want)
            for (int e = threadIdx.x; e < hh; e += kKdThreads)
                sG[(e / h) * ld + e % h] = blocks[(want ? KdHalf::kG : KdHalf::kB) * hh + e];
        held = want;
        for (int e = threadIdx.x; e < 2 * hh; e += kKdThreads) sL[(e / h) * ld + e % h] = Wi[(long long)(e / h) * nv + e % h];
        __syncthreads();
#pragma unroll
        for (int half = 0; half < 2; ++half) {
            T acc[RA][RA];
#pragma unroll
            for (int a = 0; a < RA; ++a)
#pragma unroll
                for (int b = 0; b < RA; ++b) acc[a][b] = T(0);
            const bool zero = half == 0 ? i == nn - 1 : (i == 0 || i == nn - 1);
            if (!zero) kd_product<T, RA>(acc, sL + half * h * ld, sG, h, ld, tx, ty);
#pragma unroll
            for (int a = 0; a < RA; ++a)
#pragma unroll
                for (int b = 0; b < RA; ++b) {
                    const int r = ty + 16 * a, c = tx + 16 * b;
                    if (r >= h || c >= h) continue;
                    T w = -acc[a][b];
                    if (half) w += i > 0 ? blocks[KdHalf::kDinv * hh + r * h + c] : (r == c ? T(1) : T(0));
                    Wi[(long long)(half * h + r) * nv + h + c] = w;
                }
        }
    }
}

__device__ __forceinline__ double kd_max_block(double x, double* red) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x = fmax(x, __shfl_xor_sync(0xffffffffu, x, o));
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lane == 0) red[warp] = x;
    __syncthreads();
    double t = (lane < (int)(blockDim.x >> 5)) ? red[lane] : 0.0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t = fmax(t, __shfl_xor_sync(0xffffffffu, t, o));
    __syncthreads();
    return t;
}

// Incoming datum of sample s, velocity l: entries 0..n_v/2-1 of the patch's data
// are the positive velocities at X0 (ascending), n_v/2.. the negative ones at X1.
__device__ __forceinline__ double kd_datum(const KdArgs& A, int m, int s, int l, double vl) {
    const int nv = A.n_v;
    const int t = (vl > 0.0) ? l - nv / 2 : nv / 2 + l;
    const double2 z = gaussian_pair(A.seed, (uint32_t)(t >> 1), (uint32_t)s, (uint32_t)m, kTagKinetic);
    return (t & 1) ? z.y : z.x;
}

// One CTA per (patch, kKdG samples); half-warp h owns the velocity rows h + 16 j (j < RJ),
// lane of the half = sample, so that an FP64 instruction (as long for 16 lanes as for 32)
// carries two rows and a patch spreads over twice as many CTAs: with 32 samples each the
// 192 CTAs of 64 patches x 96 samples gave 40 of 152 SMs two and the others one (8193
// nodes, 64 velocities: offline + online 127.4 ms, now 114.2; the solves 35.6 ms with the chunks
// in a second grid dimension, 29.3 in most runs numbered in one and 35.6 in the others, by how
// the 384 CTAs land on the SMs).  y (in T) shares the f layout: [node][velocity][sample]; it
// holds the residual after the residual sweep and y_i after the forward sweep.
template <class T, int RJ>
__global__ void __launch_bounds__(kKdThreads) kd_solve_kernel(KdArgs A, int M, const T* W, T* y) {
    extern __shared__ __align__(16) unsigned char kd_dyn[];
    __shared__ double red[32];
    __shared__ double c_v[kKdMaxNv], c_a[kKdMaxNv], c_d[kKdMaxNv];
    const int nv = A.n_v, chunk = blockIdx.x / M, m = blockIdx.x - chunk * M;   // patch fastest
    const int lane = threadIdx.x & (kKdG - 1), half = threadIdx.x / kKdG;
    const KPatchDev P = A.patches[m];
    const int nn = P.X1 - P.X0 + 1;
    const int s = chunk * kKdG + lane;
    const bool live = s < A.S;
    const long long n2 = (long long)nv * nv, S = A.S;
    const long long base = A.node_off[m];
    const T* Wm = W + base * n2;
    double* Fw = reinterpret_cast<double*>(kd_dyn);                 // 3 x nv x kKdLd (FP64 window)
    T* Z = reinterpret_cast<T*>(Fw + 3 * nv * kKdLd);               // nv x kKdLd (matvec input)
    const double dx = 1.0 / A.N, ie = 1.0 / A.eps;
    for (int l = threadIdx.x; l < nv; l += blockDim.x) {
        c_v[l] = A.v[l];
        c_a[l] = fabs(A.v[l]) / dx;
        c_d[l] = c_a[l] + ie * A.sigma[l];
    }
    __syncthreads();
    auto fidx = [&](int i, int l) { return ((base + i) * nv + l) * S + s; };
    const int nneg = nv / 2;   // velocities ascend: the first n_v/2 are negative
    int pass = 0;
    bool converged = false;
    for (;; ++pass) {
        // ---- residual sweep: r_i = b_i - (A f)_i, stored in y (rounded to T)
        double rmax = 0.0, fmx = 0.0;
        if (pass == 0) {
            // f = 0: the residual is the data at the identity rows
            for (int i = 0; i < nn; ++i) {
#pragma unroll
                for (int j = 0; j < RJ; ++j) {
                    const int l = half + kKdHalves * j;
                    if (l >= nv || !live) continue;
                    const double r = kd_identity(i, nn, c_v[l]) ? kd_datum(A, m, s, l, c_v[l]) : 0.0;
                    rmax = fmax(rmax, fabs(r));
                    y[fidx(i, l)] = (T)r;
                }
            }
        } else {
            // window slots: node q lives in slot q % 3
            auto load = [&](int node) {
                double* dst = Fw + (node % 3) * nv * kKdLd;
#pragma unroll
                for (int j = 0; j < RJ; ++j) {
                    const int l = half + kKdHalves * j;
                    if (l < nv) dst[l * kKdLd + lane] = live ? A.f[fidx(node, l)] : 0.0;
                }
            };
            load(0);
            for (int i = 0; i < nn; ++i) {
                if (i + 1 < nn) load(i + 1);
                __syncthreads();
                const double* Fi = Fw + (i % 3) * nv * kKdLd;
                const double* Fp = Fw + ((i + 2) % 3) * nv * kKdLd;   // node i-1 (unused at i = 0)
                const double* Fn = Fw + ((i + 1) % 3) * nv * kKdLd;   // node i+1 (unused at i = nn-1)
#pragma unroll
                for (int j = 0; j < RJ; ++j) {
                    const int l = half + kKdHalves * j;
                    if (l >= nv) continue;
                    const double vl = c_v[l], fi = Fi[l * kKdLd + lane];
                    double r, scale;
                    if (kd_identity(i, nn, vl)) {
                        r = (live ? kd_datum(A, m, s, l, vl) : 0.0) - fi;
                        scale = 1.0;
                    } else {
                        const double* kr = A.Kw + (long long)l * nv;
                        double g0 = 0.0, g1 = 0.0;
                        int k = 0;
                        for (; k + 1 < nv; k += 2) {
                            g0 = fma(__ldg(kr + k), Fi[k * kKdLd + lane], g0);
                            g1 = fma(__ldg(kr + k + 1), Fi[(k + 1) * kKdLd + lane], g1);
                        }
                        if (k < nv) g0 = fma(__ldg(kr + k), Fi[k * kKdLd + lane], g0);
                        const double nb = vl > 0.0 ? Fp[l * kKdLd + lane] : Fn[l * kKdLd + lane];
                        r = -(c_d[l] * fi - ie * (g0 + g1) - c_a[l] * nb);
                        scale = 1.0 / c_d[l];
                    }
                    if (live) {
                        rmax = fmax(rmax, fabs(r) * scale);
                        fmx = fmax(fmx, fabs(fi));
                        y[fidx(i, l)] = (T)r;
                    }
                }
                __syncthreads();   // the slot of node i-1 is reloaded with node i+2 next
            }
        }
        rmax = kd_max_block(rmax, red);
        fmx = kd_max_block(fmx, red);
        if ((pass > 0 && rmax <= A.tol * fmx) || rmax == 0.0) {   // rmax = 0: zero data, f = 0
            converged = true;
            break;
        }
        if (pass >= A.max_passes) break;
        // ---- forward sweep: y_i = W_i (r_i + a_+ y_{i-1}[+])
        T yprev[RJ];
#pragma unroll
        for (int j = 0; j < RJ; ++j) yprev[j] = T(0);
        for (int i = 0; i < nn; ++i) {
#pragma unroll
            for (int j = 0; j < RJ; ++j) {
                const int l = half + kKdHalves * j;
                if (l >= nv) continue;
                T z = live ? y[fidx(i, l)] : T(0);
                if (i > 0 && c_v[l] > 0.0) z += (T)c_a[l] * yprev[j];
                Z[l * kKdLd + lane] = z;
            }
            __syncthreads();
            const T* Wi = Wm + (long long)i * n2;
            T acc[RJ];
#pragma unroll
            for (int j = 0; j < RJ; ++j) acc[j] = T(0);
            for (int k = 0; k < nv; ++k) {
                const T zk = Z[k * kKdLd + lane];
#pragma unroll
                for (int j = 0; j < RJ; ++j) {
                    const int l = half + kKdHalves * j;
                    if (l < nv) acc[j] += __ldg(Wi + (long long)l * nv + k) * zk;
                }
            }
#pragma unroll
            for (int j = 0; j < RJ; ++j) {
                const int l = half + kKdHalves * j;
                if (l >= nv) continue;
                yprev[j] = acc[j];
                if (live) y[fidx(i, l)] = acc[j];
            }
            __syncthreads();   // Z is rewritten for the next node
        }
        // ---- backward sweep: x_i = y_i + W_i[:, -] (a_- x_{i+1}[-]); f += x
        T xnext[RJ];
#pragma unroll
        for (int j = 0; j < RJ; ++j) xnext[j] = T(0);
        for (int i = nn - 1; i >= 0; --i) {
            T x[RJ];
#pragma unroll
            for (int j = 0; j < RJ; ++j) x[j] = T(0);
            if (i < nn - 1) {
#pragma unroll
                for (int j = 0; j < RJ; ++j) {
                    const int l = half + kKdHalves * j;
                    if (l < nneg) Z[l * kKdLd + lane] = (T)c_a[l] * xnext[j];
                }
                __syncthreads();
                const T* Wi = Wm + (long long)i * n2;
                for (int k = 0; k < nneg; ++k) {
                    const T zk = Z[k * kKdLd + lane];
#pragma unroll
                    for (int j = 0; j < RJ; ++j) {
                        const int l = half + kKdHalves * j;
                        if (l < nv) x[j] += __ldg(Wi + (long long)l * nv + k) * zk;
                    }
                }
                __syncthreads();
            }
#pragma unroll
            for (int j = 0; j < RJ; ++j) {
                const int l = half + kKdHalves * j;
                if (l >= nv) continue;
                if (live) {
                    const long long q = fidx(i, l);
                    x[j] += y[q];
                    A.f[q] = (pass == 0) ? (double)x[j] : A.f[q] + (double)x[j];
                }
                xnext[j] = x[j];
            }
        }
        __syncthreads();
    }
    // restriction to K_m: node-major, velocity fastest, one sample per column
    const int i0 = P.x0 - P.X0, nk_nodes = P.x1 - P.x0 + 1;
    if (live) {
        double* out = A.snaps + P.snap_offset + (long long)s * P.n_k;
        for (int i = 0; i < nk_nodes; ++i) {
#pragma unroll
            for (int j = 0; j < RJ; ++j) {
                const int l = half + kKdHalves * j;
                if (l < nv) out[(long long)i * nv + l] = A.f[fidx(i0 + i, l)];
            }
        }
        if (half == 0) {
            A.stats[2 * ((long long)m * A.S + s) + 0] = pass;
            A.stats[2 * ((long long)m * A.S + s) + 1] = converged ? 0 : 1;
        }
    }
}

template <class T, int RA>
msp_status launch_factor(const KdArgs& A, int M, int max_nn, T* blocks, T* W, cudaStream_t s) {
    const int h = A.n_v / 2;
    const size_t tile = sizeof(T) * h * (h + 1);
    MSP_TRY(allow_smem(kd_chain_kernel<T, RA>, 4 * tile));
    MSP_TRY(allow_smem(kd_columns_kernel<T, RA>, 3 * tile));
    kd_blocks_kernel<T><<<1, 1024, sizeof(double) * h * h, s>>>(A, blocks);
    MSP_CUDA(cudaGetLastError());
    kd_chain_kernel<T, RA><<<M, kKdThreads, 4 * tile, s>>>(A, blocks, W);
    MSP_CUDA(cudaGetLastError());
    // about eight CTAs per SM over all patches
    const int per = std::max(1, std::min(max_nn, (8 * num_sms() + M - 1) / M));
    kd_columns_kernel<T, RA><<<M * per, kKdThreads, 3 * tile, s>>>(A, blocks, W, per);
    MSP_CUDA(cudaGetLastError());
    count_launches(3);
    return MSP_OK;
}

template <class T>
msp_status factor(const KMedium& K, const KdArgs& A, DevBuf<T>& blocks, T* W, cudaStream_t s) {
    const int h = A.n_v / 2;
    int max_nn = 1;
    for (auto& P : K.patches) max_nn = std::max(max_nn, P.nn);
    MSP_TRY(blocks.alloc((size_t)KdHalf::kCount * h * h, s));
    if (h <= 16) return launch_factor<T, 1>(A, K.M, max_nn, blocks.p, W, s);
    if (h <= 32) return launch_factor<T, 2>(A, K.M, max_nn, blocks.p, W, s);
    return launch_factor<T, 4>(A, K.M, max_nn, blocks.p, W, s);
}

template <class T, int RJ>
msp_status launch_solve(const KdArgs& A, int M, const T* W, T* y, cudaStream_t s) {
    const size_t smem = sizeof(double) * 3 * A.n_v * kKdLd + sizeof(T) * A.n_v * kKdLd;
    MSP_TRY(allow_smem(kd_solve_kernel<T, RJ>, smem));
    // M x chunks CTAs: the iterate alone, 32 bytes or more a (patch, sample), keeps them below 2^31
    kd_solve_kernel<T, RJ><<<M * ((A.S + kKdG - 1) / kKdG), kKdThreads, smem, s>>>(A, M, W, y);
    count_launches(1);
    MSP_CUDA(cudaGetLastError());
    return MSP_OK;
}

template <class T>
msp_status solve(const KdArgs& A, int M, const T* W, T* y, cudaStream_t s) {
    const int nv = A.n_v;
    if (nv <= 16) return launch_solve<T, 1>(A, M, W, y, s);
    if (nv <= 32) return launch_solve<T, 2>(A, M, W, y, s);
    if (nv <= 64) return launch_solve<T, 4>(A, M, W, y, s);
    return launch_solve<T, 8>(A, M, W, y, s);
}

}  // namespace

msp_status kinetic_direct_sample(KMedium& K, uint64_t seed, bool mixed, double tol, int max_iter, cudaStream_t s) {
    if (K.n_v > kKdMaxNv) {
        set_error("kinetic direct solver: at most 128 velocities");
        return MSP_ERR_INVALID_ARG;
    }
    KDirect& D = K.D;
    if (D.node_off.empty()) {
        long long off = 0;
        for (auto& P : K.patches) {
            D.node_off.push_back(off);
            off += P.nn;
        }
        D.n_nodes = off;
        MSP_TRY(upload(D.d_node_off, D.node_off, s));
    }
    const size_t n2 = (size_t)K.n_v * K.n_v;
    const size_t nf = (size_t)D.n_nodes * K.n_v * K.S;
    KdArgs A{};
    A.N = K.N; A.n_v = K.n_v; A.S = K.S;
    A.max_passes = std::max(1, std::min(max_iter, kKdMaxPasses));
    A.eps = K.eps; A.tol = tol; A.seed = seed;
    A.v = K.d_v.p; A.Kw = K.d_Kw.p; A.sigma = K.d_sigma.p; A.patches = K.d_patches.p;
    A.node_off = D.d_node_off.p;
    A.snaps = K.snaps.p; A.stats = K.stats.p;
    if (D.f.n < nf) MSP_TRY(D.f.alloc(nf, s));
    A.f = D.f.p;
    if (mixed) {
        if (!D.factored32) {
            MSP_TRY(D.W32.alloc((size_t)D.n_nodes * n2, s));
            MSP_TRY(factor<float>(K, A, D.blocks32, D.W32.p, s));
            D.factored32 = true;
        }
        if (D.y32.n < nf) MSP_TRY(D.y32.alloc(nf, s));
        return solve<float>(A, K.M, D.W32.p, D.y32.p, s);
    }
    if (!D.factored64) {
        MSP_TRY(D.W64.alloc((size_t)D.n_nodes * n2, s));
        MSP_TRY(factor<double>(K, A, D.blocks64, D.W64.p, s));
        D.factored64 = true;
    }
    if (D.y64.n < nf) MSP_TRY(D.y64.alloc(nf, s));
    return solve<double>(A, K.M, D.W64.p, D.y64.p, s);
}

}  // namespace msp
