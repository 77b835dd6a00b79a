// Per-patch Cholesky factors and their inverses (the QR remark of Sec. 3.3; the patch
// blocks of the online normal matrix), pivoted QR and Jacobi sweeps: on thread-block
// clusters where one CTA per patch would leave the GPU waiting, else one CTA per patch.
//
// A patch on the domain boundary has more than twice the snapshot columns of an inner
// one (289 against 128 on the 64-cell partitions: the boundary deltas), twelve times
// its arithmetic, so with few patches one CTA each runs for as long as the corner patch
// takes on one SM out of 152.
#include "patch_dense.h"
#include "device_util.cuh"

#include <algorithm>
#include <cmath>
#include <cooperative_groups.h>
#include <functional>
#include <queue>
#include <utility>

namespace cg = cooperative_groups;

namespace msp {

namespace {

constexpr int kPan = 16;            // columns per Cholesky panel
constexpr int kCholThreads = 512;

// Doubles of the panels p = rank, rank + nc, ... of an order-c block: rows 16 p .. c of
// 16 columns each
__host__ __device__ inline size_t panel_elems(int c, int rank, int nc) {
    size_t n = 0;
    for (int p = rank; p * kPan < c; p += nc) n += (size_t)kPan * (c - p * kPan);
    return n;
}

// Right-looking Cholesky by panels of 16 columns, dealt to the CTAs of the cluster
// panel-cyclically and held in shared memory (or in L itself, in_smem = 0).  The owner
// factors a panel and stores it to L; after a cluster barrier every CTA stages it and
// updates its own later panels.  Every element takes its updates in ascending order
// of the pivot, one FMA each, so the factor does not depend on the panel width or the
// number of CTAs.  Bound: the chain of panels and its barriers on clusters (64 patches of 128 to
// 289 columns: 1.0 ms a try, FP64 pipe busy 18% of the time, a warp waits 84 issue slots at
// barriers for each of its own), the FP64 pipe and the chain on one CTA each (1024 patches:
// 2.3 ms, 62%).  Those 64 patches took 14.4 ms with the inverse on a CTA per patch.
__global__ void __launch_bounds__(kCholThreads) patch_chol_kernel(const PatchBlock* blocks, const double* G, double* L,
                                                                  const double* shift_scale, int shifted, int* status,
                                                                  int in_smem) {
    extern __shared__ __align__(16) double csm[];
    __shared__ double s_trace;
    // Set by the owner of a panel with a bad pivot, in every CTA, by panel parity: a thread reads
    // panel p's flag after the barrier that ends the panel, while the owner of panel p + 1 may
    // already store its own; the next store to the same word, panel p + 2's, comes only after a
    // barrier that waits for every reader.
    __shared__ int s_bad[2];
    __shared__ int s_ok;
    cg::cluster_group cl = cg::this_cluster();
    const int nc = (int)cl.num_blocks(), rank = (int)cl.block_rank();
    const PatchBlock P = blocks[blockIdx.x / nc];
    const int c = P.c, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = blockDim.x >> 5;
    if (c <= 0) return;              // the whole cluster
    const double* g = G + P.off;
    double* l = L + P.off;
    double* buf = csm;               // kPan x c: the staged panel
    double* own = csm + (size_t)kPan * c;
    // column j of panel p, row i at col(p, slot)[i] (i >= 16 p)
    auto panel = [&](int p, size_t at) { return in_smem ? own + at - (size_t)p * kPan : l + (size_t)p * kPan * c; };
    auto ldp = [&](int p) { return in_smem ? (size_t)(c - p * kPan) : (size_t)c; };
    for (int i = tid; i < c; i += blockDim.x) buf[i] = g[i + (size_t)i * c];
    if (tid < 2) s_bad[tid] = 0;
    __syncthreads();
    if (tid == 0) {
        double t = 0.0;
        for (int i = 0; i < c; ++i) t += buf[i];
        s_trace = t;
    }
    cl.sync();                       // every CTA runs, and its flags are clear, before one may set them
    const double trace = s_trace;
    double shift = 0.0;
    if (shifted) shift = shift_scale[P.idx] * trace;
    int tries = 0;
    bool ok = false;
    for (; tries < 6 && !ok; ++tries) {
        size_t at = 0;
        for (int p = rank; p * kPan < c; p += nc) {
            double* pp = panel(p, at);
            const size_t ld = ldp(p);
            const int w = min(kPan, c - p * kPan);
            for (int jj = warp; jj < w; jj += nw) {
                const int j = p * kPan + jj;
                for (int i = j + lane; i < c; i += 32) pp[(size_t)jj * ld + i] = g[i + (size_t)j * c] + (i == j ? shift : 0.0);
            }
            at += (size_t)kPan * (c - p * kPan);
        }
        __syncthreads();
        ok = true;
        size_t at_next = 0;          // first of this CTA's panels not yet factored
        for (int p = 0; p * kPan < c; ++p) {
            const int k0 = p * kPan, w = min(kPan, c - k0);
            if (p % nc == rank) {
                double* pp = panel(p, at_next);
                const size_t ld = ldp(p);
                for (int k = 0; k < w; ++k) {
                    double* lk = pp + (size_t)k * ld;
                    const int kk = k0 + k;
                    if (tid == 0) {
                        const double d = lk[kk];
                        s_ok = (d > 0.0 && isfinite(d)) ? 1 : 0;
                        if (s_ok) lk[kk] = sqrt(d);
                    }
                    __syncthreads();
                    if (!s_ok) break;
                    const double piv = lk[kk];
                    for (int i = kk + 1 + tid; i < c; i += blockDim.x) lk[i] /= piv;
                    __syncthreads();
                    for (int j = k + 1 + warp; j < w; j += nw) {
                        double* lj = pp + (size_t)j * ld;
                        const double ljk = lk[k0 + j];
                        for (int i = k0 + j + lane; i < c; i += 32) lj[i] -= lk[i] * ljk;
                    }
                    __syncthreads();
                }
                if (s_ok) {
                    if (in_smem)
                        for (int jj = warp; jj < w; jj += nw)
                            for (int i = k0 + jj + lane; i < c; i += 32) __stcg(l + i + (size_t)(k0 + jj) * c, pp[(size_t)jj * ld + i]);
                } else if (tid < nc) {
                    cl.map_shared_rank(s_bad, tid)[p & 1] = 1;
                }
                at_next += (size_t)kPan * (c - k0);
                __threadfence();
            }
            cl.sync();
            if (s_bad[p & 1]) { ok = false; break; }
            const int r0 = k0 + w;
            if (r0 >= c) break;
            for (int k = warp; k < w; k += nw)
                for (int i = r0 + lane; i < c; i += 32) buf[(size_t)k * c + i] = __ldcg(l + i + (size_t)(k0 + k) * c);
            __syncthreads();
            // later panels of this CTA, a warp per column
            size_t q_at = at_next;
            int first = rank;
            while (first <= p) first += nc;
            for (int q = first; q * kPan < c; q += nc) {
                double* pq = panel(q, q_at);
                const size_t ld = ldp(q);
                const int wq = min(kPan, c - q * kPan);
                for (int jj = warp; jj < wq; jj += nw) {
                    const int j = q * kPan + jj;
                    double lj[kPan];
#pragma unroll
                    for (int k = 0; k < kPan; ++k) lj[k] = k < w ? buf[(size_t)k * c + j] : 0.0;
                    for (int i = j + lane; i < c; i += 32) {
                        double a = pq[(size_t)jj * ld + i];
#pragma unroll
                        for (int k = 0; k < kPan; ++k) a -= buf[(size_t)k * c + i] * lj[k];   // w = 16 while panels follow
                        pq[(size_t)jj * ld + i] = a;
                    }
                }
                q_at += (size_t)kPan * (c - q * kPan);
            }
            __syncthreads();
        }
        if (!ok) {
            shift = (shift == 0.0) ? 1e-14 * trace : shift * 100.0;
            cl.sync();               // every CTA has read its flag
            if (tid < 2) s_bad[tid] = 0;
            cl.sync();
        }
    }
    if (rank == 0 && tid == 0) status[P.idx] = ok ? tries : -1;
    cl.sync();                       // no CTA leaves while another may write its flags
}

// Sums over the warp of four values per lane: the lanes with (lane >> 3 & 3) == c get
// column c's.  Each value is added over the lanes in the tree of warp_sum (16, 8, ... 1),
// but with the first two levels shared, 6 additions and shuffles instead of 20.
__device__ __forceinline__ double warp_sum4(const double (&a)[4], int lane) {
    const bool hi = lane & 16, odd = lane & 8;
    double u = (hi ? a[2] : a[0]) + __shfl_xor_sync(0xffffffffu, hi ? a[0] : a[2], 16);
    double w = (hi ? a[3] : a[1]) + __shfl_xor_sync(0xffffffffu, hi ? a[1] : a[3], 16);
    double v = (odd ? w : u) + __shfl_xor_sync(0xffffffffu, odd ? u : w, 8);
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// F = L^T and Fi = L^{-T}.  X = L^{-1} column by column: X(i, j) = (delta_ij - sum_{q < i}
// l_iq X(q, j)) / l_ii, CPW columns per warp with lanes along q (q = j + lane + 32 u) and
// the partial sums combined by shuffles.  The columns of a CTA share the rows of L they
// stage in shared memory, tr rows at a time, and the reciprocals of their diagonal, one
// division per row and CTA (it takes as long as six FMAs).  X(i, j) is stored at Fi(j, i);
// the CTA of the first columns also writes F.  Columns are independent, so a patch takes
// c / kCols CTAs, and a column's sums do not depend on CPW.
// Bound by FP64 issue (pipe busy 80% of the time): 1024 patches of 128 to 289 columns 2.9 ms a
// call, 9.5 with a division per row and column and one column per warp; a 513^2 extraction went
// from 115.8 to 104.4 ms with both changes, a 2049^2 step from 1121 to 1100.
template <int CPW>
struct InvShape {
    static constexpr int kWarps = CPW == 1 ? 16 : 8;
    static constexpr int kCols = CPW * kWarps;
};

template <int CPW>
__global__ void __launch_bounds__(32 * InvShape<CPW>::kWarps) patch_inverse_kernel(const PatchBlock* blocks, const double* L,
                                                                                   double* F, double* Fi,
                                                                                   const int* status, int tr) {
    constexpr int kWarps = InvShape<CPW>::kWarps, kCols = InvShape<CPW>::kCols;
    static_assert(CPW == 1 || CPW == 4, "");
    extern __shared__ __align__(16) double ism[];
    const PatchBlock P = blocks[blockIdx.y];
    const int c = P.c, j0 = blockIdx.x * kCols;
    if (j0 >= c || (status && status[P.idx] < 0)) return;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int jb = j0 + CPW * warp;                    // the warp's first column
    const int mine = CPW == 1 ? 0 : (lane >> 3) & 3;   // the column whose sum this lane gets
    const bool writes = CPW == 1 ? lane == 0 : (lane & 7) == 0;
    const int jm = jb + mine;
    const double* l = L + P.off;
    double* f = F + P.off;
    double* fi = Fi + P.off;
    double* Ls = ism;                                  // tr x c: rows of L
    double* out = Ls + (size_t)tr * c;                 // tr x kCols
    double* rl = out + tr * kCols;                     // 1 / l_ii of the rows
    double* x = rl + tr + (size_t)CPW * warp * c;      // X(:, jb ..)
    for (int i0 = 0; i0 < c; i0 += tr) {
        const int rows = min(tr, c - i0);
        const bool live = i0 + rows > j0;              // rows above the CTA's columns hold zeros
        if (live || blockIdx.x == 0) {
            if (tid < rows) rl[tid] = 1.0 / l[(size_t)(i0 + tid) * (c + 1)];
            for (int e = tid; e < tr * (i0 + rows); e += blockDim.x) {
                const int r = e % tr, q = e / tr;
                if (r < rows) Ls[(size_t)r * c + q] = q <= i0 + r ? l[i0 + r + (size_t)q * c] : 0.0;
            }
            __syncthreads();
        }
        if (live && jb < c) {
            for (int r = 0; r < rows; ++r) {
                const int i = i0 + r;
                double v = 0.0;
                if (i >= jb) {
                    const double* li = Ls + (size_t)r * c;
                    double a[CPW];
#pragma unroll
                    for (int k = 0; k < CPW; ++k) a[k] = 0.0;
                    for (int q = jb + lane; q < i; q += 32)
#pragma unroll
                        for (int k = 0; k < CPW; ++k)
                            if (q + k < i) a[k] += li[q + k] * x[(size_t)k * c + q + k];
                    double s;
                    if constexpr (CPW == 1) s = warp_sum(a[0]);
                    else s = warp_sum4(a, lane);
                    if (i >= jm) {
                        v = ((i == jm ? 1.0 : 0.0) - s) * rl[r];
                        if (writes) x[(size_t)mine * c + i] = v;
                    }
                    __syncwarp();
                }
                if (writes) out[r * kCols + CPW * warp + mine] = v;
            }
        }
        if (blockIdx.x == 0 && F)
            for (int r = warp; r < rows; r += kWarps)
                for (int q = lane; q < c; q += 32) f[q + (size_t)(i0 + r) * c] = q <= i0 + r ? Ls[(size_t)r * c + q] : 0.0;
        __syncthreads();
        for (int e = tid; e < rows * kCols; e += blockDim.x) {
            const int r = e / kCols, w = e % kCols;
            if (j0 + w < c) fi[j0 + w + (size_t)(i0 + r) * c] = live ? out[e] : 0.0;
        }
        __syncthreads();
    }
}

// ------------------------------------------------------------------ pivoted QR
constexpr int kQrThreads = 512;
constexpr int kFormWarps = 8;       // columns of Q per CTA

// Householder QR with column pivoting of T (c x c), one patch per cluster: column r lives
// with CTA r mod nc, in shared memory (or in R, in_smem = 0).  Step j: the CTAs publish
// their largest remaining partial norm, every CTA picks the same pivot, its owner forms
// the reflector H_j = I - tau v v^T (v_0 = 1) that maps the column onto R(j, j) e_0 and
// sends v to all, and every CTA applies it to its remaining columns; the squared norms over
// the rows below are summed afresh in the same pass (no downdating).  Columns are not
// moved: a table holds the column at each position of the permuted order.
// W = R^T (lower triangular); R holds the reflectors, v below the diagonal and tau on it,
// for patch_form_q_kernel.  Bound: two cluster barriers a step and the FP64 pipe (busy 50% of
// the time).  64 patches of 128 to 289 columns: 6.2 ms and 1.6 for Q (65%), where a CTA per
// patch takes 26.
struct QrShared {
    double cand[2][kPatchCluster];   // published candidates, by step parity
    int cand_pos[2][kPatchCluster];
    double tau[2], xn2;
};

__host__ __device__ inline size_t qr_head(int c, int nc) {   // bytes before the columns
    const size_t l = (size_t)(c + nc - 1) / nc;
    return ((2 * (size_t)c + l) * sizeof(double) + (l + (size_t)c) * sizeof(int) + 15) / 16 * 16;
}

__global__ void __launch_bounds__(kQrThreads) patch_qrcp_kernel(const PatchBlock* blocks, const double* T, double* W,
                                                                double* R, double* cols, int in_smem) {
    extern __shared__ __align__(16) double qsm[];
    __shared__ QrShared S;
    cg::cluster_group cl = cg::this_cluster();
    const int nc = (int)cl.num_blocks(), rank = (int)cl.block_rank();
    const PatchBlock P = blocks[blockIdx.x / nc];
    const int c = P.c, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = blockDim.x >> 5;
    if (c < 1) return;                                       // the whole cluster
    const int nl = (c - rank + nc - 1) / nc, ml = (c + nc - 1) / nc;   // local columns
    const int lda = c | 1;
    double* vb = qsm;                                        // two reflectors, by step parity
    double* nrm = vb + 2 * (size_t)c;                        // partial norms, < 0 when taken
    int* pos = reinterpret_cast<int*>(nrm + ml);             // position of a local column
    int* perm = pos + ml;                                    // column at a position
    double* A = reinterpret_cast<double*>(reinterpret_cast<char*>(qsm) + qr_head(c, nc));
    auto col = [&](int l) { return in_smem ? A + (size_t)l * lda : cols + P.off + (size_t)(rank + l * nc) * c; };
    const double* Tm = T + P.off;
    double* Rm = R + P.off;
    for (int i = tid; i < c; i += blockDim.x) perm[i] = i;
    for (int l = warp; l < nl; l += nw) {
        double* a = col(l);
        const double* src = Tm + (size_t)(rank + l * nc) * c;
        double s = 0.0;
        for (int i = lane; i < c; i += 32) {
            const double x = src[i];
            a[i] = x;
            s = fma(x, x, s);
        }
        s = warp_sum(s);
        if (lane == 0) {
            nrm[l] = s;
            pos[l] = rank + l * nc;
        }
    }
    cl.sync();   // every CTA runs before its shared memory is written to
    for (int j = 0; j < c; ++j) {
        const int par = j & 1;
        if (warp == 0) {                                     // local candidate, to every CTA
            double best = -1.0;
            int bp = c;
            for (int l = lane; l < nl; l += 32) {
                const double x = nrm[l];
                if (x > best || (x == best && x >= 0.0 && pos[l] < bp)) { best = x; bp = pos[l]; }
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                const double ob = __shfl_xor_sync(0xffffffffu, best, o);
                const int op = __shfl_xor_sync(0xffffffffu, bp, o);
                if (ob > best || (ob == best && op < bp)) { best = ob; bp = op; }
            }
            if (lane < nc) {
                QrShared* to = cl.map_shared_rank(&S, lane);
                to->cand[par][rank] = best;
                to->cand_pos[par][rank] = bp;
            }
        }
        cl.sync();
        double best = -1.0;
        int bp = j;                                          // no candidate (NaN): the column in place
        for (int q = 0; q < nc; ++q) {
            const double b = S.cand[par][q];
            const int p = S.cand_pos[par][q];
            if (p < c && (b > best || (b == best && p < bp))) { best = b; bp = p; }
        }
        const int pc = perm[bp], moved = perm[j];            // pivot; the column it swaps with
        if (pc % nc == rank) {
            // beta = -sign(alpha) |x|, tau = (beta - alpha) / beta, v = x(1:) / (alpha - beta);
            // the squared norm below the diagonal is summed by itself (a difference of
            // the column norm and alpha^2 could cancel, and tau must match v)
            double* a = col(pc / nc);
            if (warp == 0) {
                double s = 0.0;
                for (int i = j + 1 + lane; i < c; i += 32) s = fma(a[i], a[i], s);
                s = warp_sum(s);
                if (lane == 0) S.xn2 = s;
            }
            __syncthreads();
            const double alpha = a[j], xn2 = S.xn2;
            double tau = 0.0, scal = 0.0, beta = alpha;
            if (xn2 > 0.0) {
                beta = -copysign(sqrt(alpha * alpha + xn2), alpha);
                tau = (beta - alpha) / beta;
                scal = 1.0 / (alpha - beta);
            }
            for (int i = j + 1 + tid; i < c; i += blockDim.x) {
                const double v = tau != 0.0 ? a[i] * scal : a[i];
                for (int q = 0; q < nc; ++q) cl.map_shared_rank(vb, q)[(size_t)par * c + i] = v;
                Rm[(size_t)j * c + i] = v;
            }
            if (tid < nc) cl.map_shared_rank(&S, tid)->tau[par] = tau;
            __syncthreads();
            if (tid == 0) {
                a[j] = beta;
                Rm[(size_t)j * c + j] = tau;
                nrm[pc / nc] = -1.0;
                pos[pc / nc] = j;
            }
        }
        cl.sync();
        if (tid == 0) {
            perm[j] = pc;
            perm[bp] = moved;
            if (moved != pc && moved % nc == rank) pos[moved / nc] = bp;
        }
        const double tau = S.tau[par];
        const double* v = vb + (size_t)par * c;
        // A(j:, l) -= tau v (v^T A(j:, l)) on the remaining local columns, a warp each
        for (int l = warp; l < nl; l += nw) {
            if (nrm[l] < 0.0) continue;
            double* a = col(l);
            double s = 0.0;
            if (tau != 0.0) {
                double t = (lane == 0) ? a[j] : 0.0;
                for (int i = j + 1 + lane; i < c; i += 32) t = fma(v[i], a[i], t);
                t = warp_sum(t) * tau;
                if (lane == 0) a[j] -= t;
                for (int i = j + 1 + lane; i < c; i += 32) {
                    const double x = fma(-t, v[i], a[i]);
                    a[i] = x;
                    s = fma(x, x, s);
                }
            } else {
                for (int i = j + 1 + lane; i < c; i += 32) s = fma(a[i], a[i], s);
            }
            s = warp_sum(s);
            if (lane == 0) nrm[l] = s;
        }
        __syncthreads();
    }
    // W(p, j) = R(j, p) for j <= p: the column at position p, transposed
    for (int l = warp; l < nl; l += nw) {
        const int p = pos[l];
        const double* a = col(l);
        for (int j = lane; j < c; j += 32) W[P.off + p + (size_t)j * c] = j <= p ? a[j] : 0.0;
    }
    cl.sync();   // no CTA leaves while another may write its shared memory
}

// Q = H_0 H_1 ... H_{c-1} from the reflectors: column k of Q takes H_k, ..., H_0 applied to
// e_k, a warp per column and every column by itself, so a patch takes c / 8 CTAs.
__global__ void __launch_bounds__(32 * kFormWarps) patch_form_q_kernel(const PatchBlock* blocks, const double* R,
                                                                       double* Q) {
    extern __shared__ __align__(16) double fsm[];
    const PatchBlock P = blocks[blockIdx.y];
    const int c = P.c, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int k = (int)(blockIdx.x * kFormWarps) + warp;
    if (k >= c) return;                                      // a whole warp; no block barrier follows
    double* q = fsm + (size_t)warp * c;
    const double* Rm = R + P.off;
    for (int i = lane; i < c; i += 32) q[i] = (i == k) ? 1.0 : 0.0;
    __syncwarp();
    for (int j = k; j >= 0; --j) {
        const double* v = Rm + (size_t)j * c;
        const double tau = v[j];
        if (tau != 0.0) {
            double t = (lane == 0) ? q[j] : 0.0;
            for (int i = j + 1 + lane; i < c; i += 32) t = fma(v[i], q[i], t);
            t = warp_sum(t) * tau;
            if (lane == 0) q[j] -= t;
            for (int i = j + 1 + lane; i < c; i += 32) q[i] = fma(-t, v[i], q[i]);
        }
        __syncwarp();
    }
    for (int i = lane; i < c; i += 32) Q[P.off + (size_t)k * c + i] = q[i];
}

// The same factorisation by one CTA per patch, with Q: the columns live in shared memory (or in
// W, orders above smem_c, which R^T overwrites at the end either way), are swapped into
// place, and the reflectors are applied to Q where they lie.  Every element takes the
// operations of the two kernels above in their order.  Bound by FP64 issue (1024 patches of 128
// to 289 columns 36 ms, pipe busy 72% of the time): what a patch has less of than on a
// cluster is SMs, so this form is for batches that keep them all busy; both
// sides' times stand at the rule in classify_patches.
constexpr int kQrMaxCols = 1024;    // the extraction's largest order
__global__ void __launch_bounds__(kQrThreads) patch_qr_one_kernel(const PatchBlock* blocks, const double* Tm, double* W,
                                                                  double* Q, int smem_c) {
    extern __shared__ __align__(16) double osm[];
    __shared__ double s_nrm[kQrMaxCols];
    __shared__ double s_tau[kQrMaxCols];
    __shared__ int s_piv;
    const PatchBlock S = blocks[blockIdx.x];
    const int c = S.c;
    if (c < 1 || c > kQrMaxCols) return;
    const bool in_smem = c <= smem_c;
    const int lda = in_smem ? c + 1 : c;
    double* a = in_smem ? osm : W + S.off;
    double* q = Q + S.off;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    for (long long e = threadIdx.x; e < (long long)c * c; e += blockDim.x) {
        const int i = (int)(e % c), j = (int)(e / c);
        a[i + (long long)j * lda] = Tm[S.off + e];
    }
    __syncthreads();
    for (int j = 0; j < c; ++j) {
        // squared norms of columns j.. over rows j..
        for (int col = j + warp; col < c; col += nw) {
            const double* ac = a + (long long)col * lda;
            double t = 0.0;
            for (int i = j + lane; i < c; i += 32) t = fma(ac[i], ac[i], t);
            t = warp_sum(t);
            if (lane == 0) s_nrm[col] = t;
        }
        __syncthreads();
        if (warp == 0) {
            double best = -1.0;
            int bi = j;
            for (int col = j + lane; col < c; col += 32)
                if (s_nrm[col] > best) { best = s_nrm[col]; bi = col; }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                const double ob = __shfl_xor_sync(0xffffffffu, best, o);
                const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
                if (ob > best || (ob == best && oi < bi)) { best = ob; bi = oi; }
            }
            if (lane == 0) s_piv = bi;
        }
        __syncthreads();
        const int p = s_piv;
        if (p != j) {
            for (int i = threadIdx.x; i < c; i += blockDim.x) {
                const double x = a[i + (long long)j * lda];
                a[i + (long long)j * lda] = a[i + (long long)p * lda];
                a[i + (long long)p * lda] = x;
            }
        }
        __syncthreads();
        // reflector of column j: beta = -sign(alpha) |x|, tau = (beta - alpha) / beta,
        // v = x(1:) / (alpha - beta) below the diagonal, R(j, j) = beta; the squared
        // norm below the diagonal is summed afresh (a difference of the column norm
        // and alpha^2 could cancel, and tau must match v for H_j to be orthogonal)
        double* aj = a + (long long)j * lda;
        if (warp == 0) {
            double t = 0.0;
            for (int i = j + 1 + lane; i < c; i += 32) t = fma(aj[i], aj[i], t);
            t = warp_sum(t);
            if (lane == 0) s_nrm[j] = t;
        }
        __syncthreads();
        const double alpha = aj[j];
        const double xn2 = s_nrm[j];
        double tau = 0.0, scal = 0.0, beta = alpha;
        if (xn2 > 0.0) {
            beta = -copysign(sqrt(alpha * alpha + xn2), alpha);
            tau = (beta - alpha) / beta;
            scal = 1.0 / (alpha - beta);
        }
        __syncthreads();
        if (tau != 0.0) {
            for (int i = j + 1 + threadIdx.x; i < c; i += blockDim.x) aj[i] *= scal;
        }
        if (threadIdx.x == 0) {
            aj[j] = beta;
            s_tau[j] = tau;
        }
        __syncthreads();
        if (tau != 0.0) {
            // A(j:, col) -= tau v (v^T A(j:, col)) for the trailing columns, a warp each
            for (int col = j + 1 + warp; col < c; col += nw) {
                double* ac = a + (long long)col * lda;
                double t = (lane == 0) ? ac[j] : 0.0;
                for (int i = j + 1 + lane; i < c; i += 32) t = fma(aj[i], ac[i], t);
                t = warp_sum(t) * tau;
                if (lane == 0) ac[j] -= t;
                for (int i = j + 1 + lane; i < c; i += 32) ac[i] = fma(-t, aj[i], ac[i]);
            }
        }
        __syncthreads();
    }
    // Q = H_0 ... H_{c-1}: from the identity, H_j applied to rows j.. of columns j..
    for (long long e = threadIdx.x; e < (long long)c * c; e += blockDim.x) {
        const int i = (int)(e % c), j = (int)(e / c);
        q[e] = (i == j) ? 1.0 : 0.0;
    }
    __syncthreads();
    for (int j = c - 1; j >= 0; --j) {
        const double tau = s_tau[j];
        if (tau != 0.0) {
            const double* aj = a + (long long)j * lda;
            for (int col = j + warp; col < c; col += nw) {
                double* qc = q + (long long)col * c;
                double t = (lane == 0) ? qc[j] : 0.0;
                for (int i = j + 1 + lane; i < c; i += 32) t = fma(aj[i], qc[i], t);
                t = warp_sum(t) * tau;
                if (lane == 0) qc[j] -= t;
                for (int i = j + 1 + lane; i < c; i += 32) qc[i] = fma(-t, aj[i], qc[i]);
            }
        }
        __syncthreads();
    }
    // W = R^T (lower triangular); in the global case R is read before W is written
    // over it, column by column of W = row by row of R, through registers
    if (in_smem) {
        for (long long e = threadIdx.x; e < (long long)c * c; e += blockDim.x) {
            const int i = (int)(e % c), j = (int)(e / c);
            W[S.off + e] = (i >= j) ? a[j + (long long)i * lda] : 0.0;
        }
    } else {
        // transpose in place: swap (i, j) and (j, i) for i > j, zero the upper part
        for (long long e = threadIdx.x; e < (long long)c * c; e += blockDim.x) {
            const int i = (int)(e % c), j = (int)(e / c);
            if (i > j) {
                const double r = a[j + (long long)i * lda];   // R(j, i), upper part
                a[i + (long long)j * lda] = r;                // W(i, j)
                a[j + (long long)i * lda] = 0.0;
            }
        }
    }
}

// ------------------------------------------------------------------ Jacobi
constexpr int kJacThreads = 256;
constexpr int kJacLanes = 8;                           // threads per column pair
constexpr int kJacPairs = kJacThreads / kJacLanes;     // pairs per CTA at most
constexpr int kJacCluster = 16;                        // CTAs of a patch at most (beyond the portable eight)
static_assert(kJacPairs == 32, "one warp takes the angles of a CTA's pairs");
constexpr size_t kJacSmem = 76 * 1024;                 // three CTAs per SM

struct JacShape {
    int m;        // pairs of a round (positions of the tournament)
    int slots;    // column slots of a CTA: its pairs' columns and two to receive into
    int ld;
    bool v_smem;  // V beside W in shared memory, else in global memory
    size_t bytes;
};

__host__ __device__ inline JacShape jac_shape(int c, int nc) {
    JacShape s;
    s.m = (c + 1) / 2;
    s.slots = 2 * ((s.m + nc - 1) / nc) + (nc > 1 ? 2 : 0);
    s.ld = c | 1;
    const size_t w = (size_t)s.slots * s.ld * sizeof(double);
    s.v_smem = 2 * w <= kJacSmem;
    s.bytes = s.v_smem ? 2 * w : w;
    return s;
}

struct JacArgs {
    const PatchBlock* blocks;
    double* W;
    double* V;
    int* sweeps_out;
    int max_sweeps;
    double tol, small_rel;
};

// One-sided (Hestenes) Jacobi on the columns of W (c x c), V accumulating the same
// rotations, one patch per cluster.  Column pairs follow the round-robin tournament:
// in round r position 0 plays (r, np - 1) and position i plays ((r + i), (r - i)) mod
// (np - 1), np = c rounded up to even.  From one round to the next the first player of
// a position comes from the position above, the second from the one below, so each
// CTA holds a range of positions, its columns in shared memory, and passes one
// column to each neighbour per round through distributed shared memory; a cluster
// barrier ends the round.  Phases of a round: groups of eight threads form a pair's
// inner products; one thread per pair decides and takes the angle; the CTA applies
// the rotations.  A column's squared norm is kept until the column is rotated.
// Skips: columns below u |W|_F are numerically zero; a pair orthogonal to the
// rounding floor of its inner product is left alone; and a pair whose columns are
// both below small_rel |W|_F (far under the truncation level) is left alone, since
// rotating it only mixes directions that are dropped.
// Every pair, sum and rotation is that of the one-CTA form (jacobi_svd_kernel), in
// the same order: the result does not depend on the cluster size.
// Bound: the FP64 pipe (3 c products and 8 c for the two rotations per pair) where three CTAs
// share an SM and hide each other's angles and barriers, the rounds' barriers where they
// do not.  1024 patches of 128 to 289 columns: 229 ms in both forms; the three launches, each
// by itself, keep the GPU's FP64 pipe busy 80% (900 inner patches), 41% and 4% (four corner
// patches) of their times, 65% of the 229 ms in which they overlap.  64 such patches took
// 201 ms with a CTA each, now 49 (10, 31 and 23%): a large patch no longer runs on one SM alone.
__global__ void __launch_bounds__(kJacThreads, 3) patch_jacobi_kernel(JacArgs A) {
    extern __shared__ __align__(16) double jsm[];
    constexpr int kSlots = 2 * kJacPairs + 2;
    __shared__ double s_red[16];
    __shared__ double2 s_ab[kJacPairs];                // squared norms, then cos and sin
    __shared__ double s_ga[kJacPairs];
    __shared__ int4 s_at[kJacPairs];                   // slots and columns of the pair (x < 0: none)
    __shared__ double s_nrm[kSlots];
    __shared__ int s_have[kSlots];                     // s_nrm is the norm of the column held
    __shared__ int s_col[kSlots];                      // column in a slot
    __shared__ short s_top[2][kJacPairs], s_bot[2][kJacPairs], s_free[2][2];   // by round parity
    __shared__ int s_rot, s_all[2][kJacCluster];
    cg::cluster_group cl = cg::this_cluster();
    const int nc = (int)cl.num_blocks(), rank = (int)cl.block_rank();
    const PatchBlock P = A.blocks[blockIdx.x / nc];
    const int c = P.c, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = blockDim.x >> 5;
    if (c <= 1) {                                      // the whole cluster
        if (rank == 0 && tid == 0) A.sweeps_out[P.idx] = 0;
        return;
    }
    const JacShape S = jac_shape(c, nc);
    const int np = c + (c & 1), m = S.m, ld = S.ld;
    const int lo = rank * m / nc, hi = (rank + 1) * m / nc, n = hi - lo;
    double* Wg = A.W + P.off;
    double* Vg = A.V + P.off;
    double* w = jsm;
    double* vs = jsm + (size_t)S.slots * ld;
    // |W|_F^2 in the order of a block of 512 threads: thread t takes the elements of
    // threads t and t + 256, the sixteen warp sums are added in order
    double fro2 = 0.0;
    {
        double a0 = 0.0, a1 = 0.0;
        const long long cc = (long long)c * c;
        for (long long e = tid; e < cc; e += 512) {
            const double x = Wg[e];
            a0 += x * x;
            if (e + 256 < cc) {
                const double y = Wg[e + 256];
                a1 += y * y;
            }
        }
        a0 = warp_sum(a0);
        a1 = warp_sum(a1);
        if (lane == 0) {
            s_red[warp] = a0;
            s_red[warp + 8] = a1;
        }
        __syncthreads();
        for (int k = 0; k < 16; ++k) fro2 += s_red[k];
    }
    // positions lo .. hi - 1 of round 0 in slots 2 i (first player) and 2 i + 1
    for (int i = tid; i < n; i += blockDim.x) {
        const int pr = lo + i;
        s_col[2 * i] = pr == 0 ? 0 : pr % (np - 1);
        s_col[2 * i + 1] = pr == 0 ? np - 1 : (np - 1 - pr) % (np - 1);
        s_top[0][i] = (short)(2 * i);
        s_bot[0][i] = (short)(2 * i + 1);
    }
    for (int i = tid; i < kSlots; i += blockDim.x) s_have[i] = 0;
    if (tid == 0) {
        s_free[0][0] = (short)(2 * n);
        s_free[0][1] = (short)(2 * n + 1);
        s_rot = 0;
    }
    __syncthreads();
    for (int k = warp; k < 2 * n; k += nw) {
        const int col = s_col[k];
        if (col >= c) continue;                        // the dummy player of an odd c
        for (int i = lane; i < c; i += 32) w[(size_t)k * ld + i] = Wg[(size_t)col * c + i];
        if (S.v_smem)
            for (int i = lane; i < c; i += 32) vs[(size_t)k * ld + i] = Vg[(size_t)col * c + i];
    }
    cl.sync();   // W is read before any CTA stores to it; every CTA runs before its slots are written to
    constexpr double u = 1.1102230246251565e-16;
    const double tol = A.tol, small_rel = A.small_rel;
    const double negligible = u * u * fro2;
    const double floor_abs = 2.0 * c * u * sqrt(fro2);
    const double small2 = small_rel * small_rel * fro2;
    const double inv_fro2 = 1.0 / fro2;
    const float floor_rel = 2.0f * c * (float)u;
    const int g = tid & (kJacLanes - 1), pr = tid / kJacLanes;
    int par = 0, sweep = 0;
    for (; sweep < A.max_sweeps; ++sweep) {
        for (int r = 0; r < np - 1; ++r) {
            // phase 1
            int kp = 0, kq = 0;
            bool real = false;
            if (pr < n) {
                kp = s_top[par][pr];
                kq = s_bot[par][pr];
                if (s_col[kp] > s_col[kq]) { const int t = kp; kp = kq; kq = t; }
                real = s_col[kq] < c;
            }
            double al = 0, be = 0, ga = 0;
            const bool have = !real || (s_have[kp] && s_have[kq]);
            if (__all_sync(0xffffffffu, have)) {
                // norms kept: the inner product alone, and not for pairs the norms already skip
                if (real) {
                    al = s_nrm[kp];
                    be = s_nrm[kq];
                }
                const bool skip = al <= negligible || be <= negligible || (al < small2 && be < small2);
                if (real && !skip) {
                    const double* wp = w + (size_t)kp * ld;
                    const double* wq = w + (size_t)kq * ld;
                    for (int i = g; i < c; i += kJacLanes) ga = fma(wp[i], wq[i], ga);
                }
#pragma unroll
                for (int o = kJacLanes / 2; o > 0; o >>= 1) ga += __shfl_xor_sync(0xffffffffu, ga, o);
            } else {
                if (real) {
                    const double* wp = w + (size_t)kp * ld;
                    const double* wq = w + (size_t)kq * ld;
                    for (int i = g; i < c; i += kJacLanes) {
                        const double x = wp[i], y = wq[i];
                        al = fma(x, x, al);
                        be = fma(y, y, be);
                        ga = fma(x, y, ga);
                    }
                }
#pragma unroll
                for (int o = kJacLanes / 2; o > 0; o >>= 1) {
                    al += __shfl_xor_sync(0xffffffffu, al, o);
                    be += __shfl_xor_sync(0xffffffffu, be, o);
                    ga += __shfl_xor_sync(0xffffffffu, ga, o);
                }
                if (real && g == 0) {
                    s_nrm[kp] = al;
                    s_nrm[kq] = be;
                    s_have[kp] = s_have[kq] = 1;
                }
            }
            if (pr < n && g == 0) {
                s_at[pr] = real ? make_int4(kp, kq, s_col[kp], s_col[kq]) : make_int4(-1, 0, 0, 0);
                s_ab[pr] = make_double2(al, be);
                s_ga[pr] = ga;
            }
            __syncthreads();
            // phase 2, by one warp, another each round (a warp's FP64 instructions all go to
            // its quarter of the SM): the decision in FP32 on values scaled by 1 / |W|_F^2
            // where it is clear by a percent, else as stated; then the angle
            if (warp == (r & (nw - 1)) && lane < n && s_at[lane].x >= 0) {
                const double a = s_ab[lane].x, b = s_ab[lane].y, gg = s_ga[lane];
                bool go = !(a <= negligible || b <= negligible || (a < small2 && b < small2));
                if (go) {
                    const float af = sqrtf((float)(a * inv_fro2)), bf = sqrtf((float)(b * inv_fro2));
                    const float gf = fabsf((float)(gg * inv_fro2));
                    const float bound = (float)tol * af * bf + floor_rel * (af + bf);
                    if (!(gf > 1.01f * bound)) {
                        if (gf < 0.99f * bound) {
                            go = false;
                        } else {
                            const double na = sqrt(a), nb = sqrt(b);
                            go = !(fabs(gg) <= tol * na * nb + floor_abs * (na + nb));
                        }
                    }
                }
                if (!go) {
                    s_at[lane].x = -1;
                } else {
                    const double zeta = (b - a) / (2.0 * gg);
                    const double t = (zeta >= 0.0 ? 1.0 : -1.0) / (fabs(zeta) + sqrt(1.0 + zeta * zeta));
                    const double cs = 1.0 / sqrt(1.0 + t * t);
                    s_ab[lane] = make_double2(cs, cs * t);
                    s_have[s_top[par][lane]] = s_have[s_bot[par][lane]] = 0;
                    s_rot = 1;
                }
            }
            __syncthreads();
            // phase 3: rows fastest over the pairs
            for (int e = tid; e < n * c; e += blockDim.x) {
                const int k = e / c, i = e - k * c;
                const int4 at = s_at[k];
                if (at.x < 0) continue;
                const double2 rot = s_ab[k];
                const double cs = rot.x, sn = rot.y;
                double xv, yv;
                double *vp, *vq;
                if (S.v_smem) {
                    vp = vs + at.x * ld + i;
                    vq = vs + at.y * ld + i;
                    xv = *vp;
                    yv = *vq;
                } else {                               // other CTAs held these columns: past the L1
                    vp = Vg + at.z * c + i;
                    vq = Vg + at.w * c + i;
                    xv = __ldcg(vp);
                    yv = __ldcg(vq);
                }
                double* xp = w + at.x * ld + i;
                double* xq = w + at.y * ld + i;
                const double x = *xp, y = *xq;
                *xp = cs * x - sn * y;
                *xq = sn * x + cs * y;
                const double rv = cs * xv - sn * yv, ru = sn * xv + cs * yv;
                if (S.v_smem) {
                    *vp = rv;
                    *vq = ru;
                } else {
                    __stcg(vp, rv);
                    __stcg(vq, ru);
                }
            }
            __syncthreads();
            // next round's positions; the columns leaving the CTA go to the slots their
            // neighbours keep free
            const int nxt = par ^ 1;
            for (int i = tid; i < n; i += blockDim.x) {
                short nt, nb;
                if (i + 1 < n) nt = s_top[par][i + 1];
                else nt = hi < m ? s_free[par][0] : s_bot[par][i];
                if (lo + i == 0) nb = s_bot[par][0];
                else if (i == 0) nb = s_free[par][1];
                else nb = lo + i == 1 ? s_top[par][0] : s_bot[par][i - 1];
                if (m == 1) { nt = s_top[par][0]; nb = s_bot[par][0]; }
                s_top[nxt][i] = nt;
                s_bot[nxt][i] = nb;
            }
            if (tid == 0) {
                s_free[nxt][0] = lo > 0 ? s_top[par][0] : s_bot[par][n - 1];
                s_free[nxt][1] = hi < m ? s_bot[par][n - 1] : s_top[par][0];
            }
            for (int dir = 0; dir < 2; ++dir) {
                if (dir == 0 ? lo == 0 : hi == m) continue;
                const int to = dir == 0 ? rank - 1 : rank + 1;
                const int k = dir == 0 ? s_top[par][0] : s_bot[par][n - 1];
                const int dst = cl.map_shared_rank(&s_free[par][0], to)[dir == 0 ? 0 : 1];
                double* rw = cl.map_shared_rank(w, to) + (size_t)dst * ld;
                const int half = blockDim.x / 2, t = tid - dir * half;
                if (t >= 0 && t < half) {
                    for (int i = t; i < c; i += half) rw[i] = w[(size_t)k * ld + i];
                    if (S.v_smem) {
                        double* rv = cl.map_shared_rank(vs, to) + (size_t)dst * ld;
                        for (int i = t; i < c; i += half) rv[i] = vs[(size_t)k * ld + i];
                    }
                    if (t == 0) {
                        cl.map_shared_rank(s_col, to)[dst] = s_col[k];
                        cl.map_shared_rank(s_nrm, to)[dst] = s_nrm[k];
                        cl.map_shared_rank(s_have, to)[dst] = s_have[k];
                    }
                }
            }
            if (r == np - 2 && tid < nc) cl.map_shared_rank(&s_all[sweep & 1][0], tid)[rank] = s_rot;
            if (nc > 1) {
                if (!S.v_smem) __threadfence();
                cl.sync();
            } else {
                __syncthreads();
            }
            par = nxt;
        }
        int rot = 0;
        for (int k = 0; k < nc; ++k) rot |= s_all[sweep & 1][k];
        if (rot == 0) break;
        if (tid == 0) s_rot = 0;     // set again only after the next round's first barrier
    }
    for (int k = warp; k < 2 * n; k += nw) {
        const int slot = (k & 1) ? s_bot[par][k >> 1] : s_top[par][k >> 1];
        const int col = s_col[slot];
        if (col >= c) continue;
        for (int i = lane; i < c; i += 32) Wg[(size_t)col * c + i] = w[(size_t)slot * ld + i];
        if (S.v_smem)
            for (int i = lane; i < c; i += 32) Vg[(size_t)col * c + i] = vs[(size_t)slot * ld + i];
    }
    if (rank == 0 && tid == 0) A.sweeps_out[P.idx] = sweep;
}

template <class... KArgs, class... Args>
msp_status launch_cluster(void (*kernel)(KArgs...), int patches, int nc, int threads, size_t smem, cudaStream_t s,
                          Args... args) {
    MSP_TRY(allow_smem(kernel, smem));
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)(patches * nc));
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = (unsigned)nc;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    MSP_CUDA(cudaLaunchKernelEx(&cfg, kernel, args...));
    count_launches(1);
    return MSP_OK;
}

// dynamic shared memory a block may ask for, less the kernels' static part
msp_status smem_room(size_t* room) {
    int dev = 0, optin = 0;
    MSP_CUDA(cudaGetDevice(&dev));
    MSP_CUDA(cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
    *room = (size_t)optin - 4096;
    return MSP_OK;
}

// Time at which the last of `jobs` (a patch's CTAs, which start together; the SM sixths that each
// takes; its time) ends when they are started in order as room on the device comes free.
struct Job {
    int ctas, sixths;
    double time;
};
double makespan(const std::vector<Job>& jobs) {
    long long room = 6LL * num_sms();
    double now = 0.0, last = 0.0;
    std::priority_queue<std::pair<double, int>, std::vector<std::pair<double, int>>, std::greater<>> running;   // end, sixths
    for (const Job& j : jobs) {
        const int need = j.ctas * j.sixths;
        while (room < need && !running.empty()) {
            now = running.top().first;
            room += running.top().second;
            running.pop();
        }
        running.push({now + j.time, need});
        room -= need;
        last = std::max(last, now + j.time);
    }
    return last;
}

}  // namespace

PatchClasses classify_patches(const std::vector<int>& cols, const std::vector<long long>& off) {
    PatchClasses C;
    double total = 0.0;
    for (int c : cols) total += (double)c * c * c;
    const double share = total / num_sms();
    std::vector<PatchBlock> small;
    for (size_t m = 0; m < cols.size(); ++m) {
        const double w = (double)cols[m] * cols[m] * cols[m];
        // candidates: the patches that alone would keep one SM for more than half of the time
        // in which the whole batch keeps all of them, and those above the order whose columns
        // one SM's shared memory holds; below 48 columns a cluster has no advantage
        const bool big = (w > 0.5 * share && cols[m] >= 48) || cols[m] > 160;
        const PatchBlock b{off[m], cols[m], (int)m};
        (big ? C.blocks : small).push_back(b);
    }
    auto larger = [](const PatchBlock& a, const PatchBlock& b) { return a.c > b.c; };
    std::stable_sort(C.blocks.begin(), C.blocks.end(), larger);
    std::stable_sort(small.begin(), small.end(), larger);
    // They take clusters, and the others one CTA each after them, if that ends before one CTA for
    // every patch does.  Times in us of the QR with Q, the longest of the stages: a patch alone
    // on one CTA and on a cluster of eight (24 to 160 columns, fitted), the latter times 1.15 for
    // the clusters beside it, two of whose CTAs share an SM.  Over 272 batches (1 to 1600 patches
    // of 20 to 373 columns) the choice takes 0.3 percent longer than the better one on average, 14 at
    // most.  Clusters against one CTA each, ms:
    //   QR and Q               64 patches of 128 to 289 columns 7.7 : 25.9, 8 of 64 0.73 : 0.97;
    //                          1024 of 128 to 289 45.8 : 36.5, 256 of 128 to 165 17.8 : 8.8, 400 of
    //                          20 to 69 2.2 : 1.2, 64 of 96 3.0 : 2.0
    //   Cholesky and inverse   64 of 128 to 289 1.6 : 2.5; 1024 of 128 to 289 6.2 : 5.0, 152 of 160
    //                          2.1 : 1.1, 64 of 96 0.52 : 0.37
    auto one = [](int c) { return Job{1, 6, c * (6.5 + c * (0.1 + c * 5.4e-4))}; };
    auto cluster = [](int c) { return Job{kPatchCluster, 3, 1.15 * c * (9.5 + c * 0.024)}; };
    std::vector<Job> with, rest, without;
    for (const PatchBlock& b : C.blocks) {
        with.push_back(cluster(b.c));
        without.push_back(one(b.c));
    }
    for (const PatchBlock& b : small) {
        rest.push_back(one(b.c));
        without.push_back(one(b.c));
    }
    if (makespan(with) + makespan(rest) >= makespan(without)) {
        C.blocks.insert(C.blocks.end(), small.begin(), small.end());
        small.swap(C.blocks);
        C.blocks.clear();
    }
    C.n_big = (int)C.blocks.size();
    if (!C.blocks.empty()) C.max_c[0] = C.blocks.front().c;
    if (!small.empty()) C.max_c[1] = small.front().c;
    C.blocks.insert(C.blocks.end(), small.begin(), small.end());
    return C;
}

template <int CPW>
static msp_status launch_inverse(const PatchClasses& C, int c, const PatchBlock* blocks, const double* L, double* F,
                                 double* Fi, const int* status, cudaStream_t s) {
    constexpr int kWarps = InvShape<CPW>::kWarps, kCols = InvShape<CPW>::kCols;
    size_t room = 0;
    MSP_TRY(smem_room(&room));
    int tr = 16;
    auto bytes = [&](int t) { return sizeof(double) * ((size_t)t * (c + kCols + 1) + (size_t)kCols * c); };
    while (tr > 1 && bytes(tr) > room) tr /= 2;
    MSP_TRY(allow_smem(patch_inverse_kernel<CPW>, bytes(tr)));
    for (size_t b0 = 0; b0 < C.blocks.size(); b0 += 65535) {
        const unsigned nb = (unsigned)std::min<size_t>(65535, C.blocks.size() - b0);
        patch_inverse_kernel<CPW><<<dim3((c + kCols - 1) / kCols, nb), 32 * kWarps, bytes(tr), s>>>(blocks + b0, L, F, Fi,
                                                                                                  status, tr);
        count_launches(1);
    }
    MSP_CUDA(cudaGetLastError());
    return MSP_OK;
}

static msp_status launch_inverse(const PatchClasses& C, const PatchBlock* blocks, const double* L, double* F, double* Fi,
                                 const int* status, cudaStream_t s) {
    const int c = std::max(C.max_c[0], C.max_c[1]);
    if (c <= 0) return MSP_OK;
    long long columns = 0;
    for (const PatchBlock& b : C.blocks) columns += b.c;
    // Four columns a warp need about 26 FP64 instructions a row where one needs 11.5, so they
    // win from about two columns per quarter of an SM on; beyond 512 columns their 32 vectors
    // would leave shared memory no room for the rows.
    const bool four = columns >= 2LL * 4 * num_sms() && c <= 512;
    return four ? launch_inverse<4>(C, c, blocks, L, F, Fi, status, s) : launch_inverse<1>(C, c, blocks, L, F, Fi, status, s);
}

msp_status patch_triangular_inverse(const PatchClasses& C, const PatchBlock* blocks, const double* L, double* Fi,
                                    cudaStream_t s) {
    return launch_inverse(C, blocks, L, nullptr, Fi, nullptr, s);
}

msp_status patch_cholesky(const PatchClasses& C, const PatchBlock* blocks, const double* G, double* L, double* F,
                          double* Fi, const double* shift_scale, bool shifted, int* status, cudaStream_t s) {
    size_t room = 0;
    MSP_TRY(smem_room(&room));
    const int count[2] = {C.n_big, (int)C.blocks.size() - C.n_big};
    for (int cls = 0; cls < 2; ++cls) {
        if (!count[cls] || C.max_c[cls] <= 0) continue;
        const int nc = cls == 0 ? kPatchCluster : 1, c = C.max_c[cls];
        const size_t head = sizeof(double) * (size_t)kPan * c, own = sizeof(double) * panel_elems(c, 0, nc);
        const int in_smem = head + own <= room ? 1 : 0;
        MSP_TRY(launch_cluster(patch_chol_kernel, count[cls], nc, kCholThreads, in_smem ? head + own : head, s,
                               blocks + (cls == 0 ? 0 : C.n_big), G, L, shift_scale, shifted ? 1 : 0, status, in_smem));
    }
    return launch_inverse(C, blocks, L, F, Fi, status, s);
}

msp_status patch_qrcp(const PatchClasses& C, const PatchBlock* blocks, const double* T, double* W, double* Q, double* R,
                      double* cols, cudaStream_t s) {
    size_t room = 0;
    MSP_TRY(smem_room(&room));
    const int c0 = C.max_c[0], n_cluster = C.n_big;
    const int n_one = (int)C.blocks.size() - n_cluster;
    if (n_cluster > 0) {
        const size_t own = sizeof(double) * ((size_t)(c0 + kPatchCluster - 1) / kPatchCluster) * (c0 | 1),
                     head = qr_head(c0, kPatchCluster);
        const int in_smem = head + own <= room ? 1 : 0;
        MSP_TRY(launch_cluster(patch_qrcp_kernel, n_cluster, kPatchCluster, kQrThreads, in_smem ? head + own : head, s,
                               blocks, T, W, R, cols, in_smem));
        const size_t bytes = sizeof(double) * (size_t)kFormWarps * c0;
        MSP_TRY(allow_smem(patch_form_q_kernel, bytes));
        for (int b0 = 0; b0 < n_cluster; b0 += 65535) {
            const unsigned nb = (unsigned)std::min(65535, n_cluster - b0);
            patch_form_q_kernel<<<dim3((c0 + kFormWarps - 1) / kFormWarps, nb), 32 * kFormWarps, bytes, s>>>(blocks + b0, R, Q);
            count_launches(1);
        }
        MSP_CUDA(cudaGetLastError());
    }
    if (n_one > 0) {
        const int c = C.max_c[1];
        cudaFuncAttributes fa{};
        MSP_CUDA(cudaFuncGetAttributes(&fa, patch_qr_one_kernel));
        room += 3072;                                        // all but the 1 KB a block reserves
        room -= fa.sharedSizeBytes;
        int cq = 0;                                          // largest order held in shared memory
        while (cq < c && (size_t)(cq + 1) * (cq + 2) * sizeof(double) <= room) ++cq;
        const size_t bytes = (size_t)cq * (cq + 1) * sizeof(double);
        MSP_TRY(allow_smem(patch_qr_one_kernel, bytes));
        patch_qr_one_kernel<<<n_one, kQrThreads, bytes, s>>>(blocks + n_cluster, T, W, Q, cq);
        count_launches(1);
        MSP_CUDA(cudaGetLastError());
    }
    return MSP_OK;
}

// Cluster sizes of the sweeps: 2, 4, 8 and 16, and two between.  5 takes the orders that four
// CTAs of 32 pairs do not hold (257 to 320 columns) without going to eight; 10 is the next
// step for a patch whose share asks for more than eight.
constexpr int kJacSizes = 7;
constexpr int kJacNc[kJacSizes] = {16, 10, 8, 5, 4, 2, 1};

// Cluster size of one patch: enough CTAs that it takes about its share of the GPU (twice
// its work over the work per SM: up to three CTAs share an SM), as far as its columns
// need them (32 pairs a CTA, W in shared memory) and as long as each has six pairs (below
// that a round is shorter than its barriers); one below 48 columns; 0 when no cluster
// holds W.
static int jac_cluster(int c, double share, size_t room, int max_nc) {
    auto fits = [&](int nc) {
        const JacShape s = jac_shape(c, nc);
        return s.bytes <= (nc > kPatchCluster ? kJacSmem : room) && (s.m + nc - 1) / nc <= kJacPairs;
    };
    if (c < 48) return fits(1) ? 1 : 0;
    const double want = 2.0 * c * c * c / share;
    int best = 0;
    for (int q = kJacSizes - 2; q >= 0; --q) {         // ascending from 2
        const int nc = kJacNc[q];
        if (nc > max_nc || (best && (c + 1) / 2 < 6 * nc)) break;
        if (!fits(nc)) continue;
        best = nc;
        if (nc >= want) break;
    }
    return best;
}

// Streams beside the caller's for launches that may overlap; on every way out the
// caller's stream waits for them.
struct ForkedStreams {
    cudaStream_t main = nullptr;
    cudaStream_t st[kJacSizes] = {};
    cudaEvent_t fork = nullptr, join[kJacSizes] = {};
    int n = 0;
    msp_status open(cudaStream_t s) {
        main = s;
        MSP_CUDA(cudaEventCreateWithFlags(&fork, cudaEventDisableTiming));
        MSP_CUDA(cudaEventRecord(fork, s));
        return MSP_OK;
    }
    msp_status next(cudaStream_t* out) {
        MSP_CUDA(cudaStreamCreateWithFlags(&st[n], cudaStreamNonBlocking));
        const int k = n++;
        MSP_CUDA(cudaEventCreateWithFlags(&join[k], cudaEventDisableTiming));
        MSP_CUDA(cudaStreamWaitEvent(st[k], fork, 0));
        *out = st[k];
        return MSP_OK;
    }
    ~ForkedStreams() {
        for (int k = 0; k < n; ++k) {
            if (join[k]) {
                cudaEventRecord(join[k], st[k]);
                cudaStreamWaitEvent(main, join[k], 0);
                cudaEventDestroy(join[k]);
            }
            cudaStreamDestroy(st[k]);                  // released when its work is done
        }
        if (fork) cudaEventDestroy(fork);
    }
};

msp_status patch_jacobi(const std::vector<PatchBlock>& all, double* W, double* V, int max_sweeps, double tol,
                        double small_rel, int* sweeps, DevBuf<PatchBlock>& d_blocks, std::vector<PatchBlock>& rest,
                        cudaStream_t s) {
    size_t room = 0;
    MSP_TRY(smem_room(&room));
    room -= 4096;                                      // the kernel's tables
    double total = 0.0;
    for (const PatchBlock& b : all) total += (double)b.c * b.c * b.c;
    const double share = total / num_sms();
    // more than 8 CTAs in a cluster are an option of the device: ask whether one can be resident
    int max_nc = kPatchCluster;
    MSP_CUDA(cudaFuncSetAttribute(patch_jacobi_kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
    MSP_TRY(allow_smem(patch_jacobi_kernel, room));
    for (int q = 0; q < kJacSizes && kJacNc[q] > max_nc; ++q) {
        cudaLaunchConfig_t cfg{};
        cfg.gridDim = dim3((unsigned)kJacNc[q]);
        cfg.blockDim = dim3(kJacThreads);
        cfg.dynamicSmemBytes = kJacSmem;
        cudaLaunchAttribute at{};
        at.id = cudaLaunchAttributeClusterDimension;
        at.val.clusterDim.x = (unsigned)kJacNc[q];
        at.val.clusterDim.y = at.val.clusterDim.z = 1;
        cfg.attrs = &at;
        cfg.numAttrs = 1;
        int clusters = 0;
        if (cudaOccupancyMaxActiveClusters(&clusters, patch_jacobi_kernel, &cfg) == cudaSuccess && clusters > 0)
            max_nc = kJacNc[q];
        else
            (void)cudaGetLastError();
    }
    std::vector<PatchBlock> list;
    rest.clear();
    int first[kJacSizes + 1] = {};
    size_t bytes[kJacSizes] = {};
    for (int q = 0; q < kJacSizes; ++q) {
        first[q] = (int)list.size();
        for (const PatchBlock& b : all) {
            const int nc = jac_cluster(b.c, share, room, max_nc);
            if (nc == kJacNc[q]) {
                list.push_back(b);
                bytes[q] = std::max(bytes[q], jac_shape(b.c, nc).bytes);
            } else if (nc == 0 && q == 0) {
                rest.push_back(b);
            }
        }
    }
    first[kJacSizes] = (int)list.size();
    // One CTA per patch (jacobi_svd_kernel) where that ends sooner.  A patch on one CTA of 16
    // warps takes about c^2.5 (the dropped columns are skipped), a CTA of a cluster, of 8 warps
    // and with a barrier per round, 2.1 c^2.5 / nc whether one, two or three share its SM.  Clusters win where patches are few or uneven, one CTA each where the
    // clusters' shared memory leaves one or two CTAs per SM or their last wave is nearly empty.
    // Sweeps on clusters against one CTA each: 64 patches of 128 to 289 columns 48.6 ms against
    // 217, 196 of 100 to 221 40.7 against 105; 196 of 200 to 253 176 against 115, 484 of 150 to 219
    // 157 against 127, 324 of 160 to 281 223 against 186.
    {
        std::vector<Job> cluster, one;
        auto work = [](int c) { return c > 1 ? (double)c * c * std::sqrt((double)c) : 0.0; };
        for (int q = 0; q < kJacSizes; ++q) {
            if (first[q] == first[q + 1]) continue;
            int per_sm = 0;
            MSP_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, patch_jacobi_kernel, kJacThreads, bytes[q]));
            per_sm = std::max(1, std::min(per_sm, 3));
            for (int k = first[q]; k < first[q + 1]; ++k)
                cluster.push_back(Job{kJacNc[q], 6 / per_sm, 2.1 * work(list[k].c) / kJacNc[q]});
        }
        for (const PatchBlock& b : rest) cluster.push_back(Job{1, 6, work(b.c)});   // they follow on one CTA
        for (const PatchBlock& b : all) one.push_back(Job{1, 6, work(b.c)});
        if (makespan(one) < makespan(cluster)) {
            rest = all;
            return MSP_OK;
        }
    }
    MSP_TRY(upload(d_blocks, list, s));
    // the largest patches first, the other sizes beside them
    ForkedStreams fs;
    MSP_TRY(fs.open(s));
    bool on_main = true;
    for (int q = 0; q < kJacSizes; ++q) {
        const int count = first[q + 1] - first[q];
        if (!count) continue;
        cudaStream_t ss = s;
        if (!on_main) MSP_TRY(fs.next(&ss));
        on_main = false;
        const JacArgs a{d_blocks.p + first[q], W, V, sweeps, max_sweeps, tol, small_rel};
        MSP_TRY(launch_cluster(patch_jacobi_kernel, count, kJacNc[q], kJacThreads, bytes[q], ss, a));
    }
    return MSP_OK;
}

}  // namespace msp
