// Per-patch Cholesky factors and their inverses (the QR remark of Sec. 3.3; the patch
// blocks of the online normal matrix), spread over the GPU by rows of work instead of
// one CTA per patch.
//
// A patch on the domain boundary has more than twice the snapshot columns of an inner
// one (289 against 128 on the 64-cell partitions: the boundary deltas), twelve times
// its arithmetic, so one CTA per patch ran for as long as the corner patch took on one
// SM out of 152, and out of global memory.
#include "patch_dense.h"
#include "device_util.cuh"

#include <algorithm>
#include <cooperative_groups.h>

namespace cg = cooperative_groups;

namespace msp {

namespace {

constexpr int kPan = 16;            // columns per Cholesky panel
constexpr int kCholThreads = 512;
constexpr int kInvWarps = 16;       // columns of the inverse per CTA

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
// number of CTAs.
__global__ void __launch_bounds__(kCholThreads) patch_chol_kernel(const PatchBlock* blocks, const double* G, double* L,
                                                                  const double* shift_scale, int shifted, int* status,
                                                                  int in_smem) {
    extern __shared__ __align__(16) double csm[];
    __shared__ double s_trace;
    __shared__ int s_bad;            // set by the owner of a panel with a bad pivot, in every CTA
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
    if (tid == 0) s_bad = 0;
    __syncthreads();
    if (tid == 0) {
        double t = 0.0;
        for (int i = 0; i < c; ++i) t += buf[i];
        s_trace = t;
    }
    cl.sync();                       // every CTA runs, and its flag is clear, before one may set it
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
                    *cl.map_shared_rank(&s_bad, tid) = 1;
                }
                at_next += (size_t)kPan * (c - k0);
                __threadfence();
            }
            cl.sync();
            if (s_bad) { ok = false; break; }
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
            if (tid == 0) s_bad = 0;
            cl.sync();
        }
    }
    if (rank == 0 && tid == 0) status[P.idx] = ok ? tries : -1;
    cl.sync();                       // no CTA leaves while another may write its flag
}

// F = L^T and Fi = L^{-T}.  X = L^{-1} column by column: X(i, j) = (delta_ij - sum_{q < i}
// l_iq X(q, j)) / l_ii, one warp per column j with lanes along q (q = j + lane + 32 u) and
// the warp's partial sums combined by shuffles, sixteen columns per CTA sharing the
// rows of L they stage in shared memory, tr rows at a time.  X(i, j) is stored at
// Fi(j, i); the CTA of the first columns also writes F.  Columns are independent, so a
// patch takes c / 16 CTAs.
__global__ void __launch_bounds__(32 * kInvWarps) patch_inverse_kernel(const PatchBlock* blocks, const double* L,
                                                                       double* F, double* Fi, const int* status,
                                                                       int tr) {
    extern __shared__ __align__(16) double ism[];
    const PatchBlock P = blocks[blockIdx.y];
    const int c = P.c, j0 = blockIdx.x * kInvWarps;
    if (j0 >= c || status[P.idx] < 0) return;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int j = j0 + warp;
    const double* l = L + P.off;
    double* f = F + P.off;
    double* fi = Fi + P.off;
    double* Ls = ism;                                  // tr x c: rows of L
    double* out = Ls + (size_t)tr * c;                 // tr x kInvWarps
    double* x = out + tr * kInvWarps + (size_t)warp * c;   // X(:, j)
    for (int i0 = 0; i0 < c; i0 += tr) {
        const int rows = min(tr, c - i0);
        const bool live = i0 + rows > j0;              // rows above the CTA's columns hold zeros
        if (live || blockIdx.x == 0) {
            for (int e = tid; e < tr * (i0 + rows); e += blockDim.x) {
                const int r = e % tr, q = e / tr;
                if (r < rows) Ls[(size_t)r * c + q] = q <= i0 + r ? l[i0 + r + (size_t)q * c] : 0.0;
            }
            __syncthreads();
        }
        if (live && j < c) {
            for (int r = 0; r < rows; ++r) {
                const int i = i0 + r;
                double v = 0.0;
                if (i >= j) {
                    const double* li = Ls + (size_t)r * c;
                    const double rli = 1.0 / li[i];
                    double a = 0.0;
                    for (int q = j + lane; q < i; q += 32) a += li[q] * x[q];
                    a = warp_sum(a);
                    v = ((i == j ? 1.0 : 0.0) - a) * rli;
                    if (lane == 0) x[i] = v;
                    __syncwarp();
                }
                if (lane == 0) out[r * kInvWarps + warp] = v;
            }
        }
        if (blockIdx.x == 0)
            for (int r = warp; r < rows; r += kInvWarps)
                for (int q = lane; q < c; q += 32) f[q + (size_t)(i0 + r) * c] = q <= i0 + r ? Ls[(size_t)r * c + q] : 0.0;
        __syncthreads();
        for (int e = tid; e < rows * kInvWarps; e += blockDim.x) {
            const int r = e / kInvWarps, w = e % kInvWarps;
            if (j0 + w < c) fi[j0 + w + (size_t)(i0 + r) * c] = live ? out[e] : 0.0;
        }
        __syncthreads();
    }
}

template <class... KArgs, class... Args>
msp_status launch_cluster(void (*kernel)(KArgs...), int patches, int nc, int threads, size_t smem, cudaStream_t s,
                          Args... args) {
    MSP_CUDA(cudaFuncSetAttribute((const void*)kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
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

}  // namespace

PatchClasses classify_patches(const std::vector<int>& cols, const std::vector<long long>& off) {
    PatchClasses C;
    double total = 0.0;
    for (int c : cols) total += (double)c * c * c;
    const double share = total / num_sms();
    std::vector<PatchBlock> small;
    for (size_t m = 0; m < cols.size(); ++m) {
        const double w = (double)cols[m] * cols[m] * cols[m];
        // A cluster for every patch that alone would keep one SM for more than half of
        // the time in which the whole batch keeps all of them, and above the order
        // whose columns one SM's shared memory holds; below 48 columns eight CTAs
        // would spend their time in barriers.
        const bool big = (w > 0.5 * share && cols[m] >= 48) || cols[m] > 160;
        const PatchBlock b{off[m], cols[m], (int)m};
        (big ? C.blocks : small).push_back(b);
    }
    auto larger = [](const PatchBlock& a, const PatchBlock& b) { return a.c > b.c; };
    std::stable_sort(C.blocks.begin(), C.blocks.end(), larger);
    std::stable_sort(small.begin(), small.end(), larger);
    C.n_big = (int)C.blocks.size();
    if (!C.blocks.empty()) C.max_c[0] = C.blocks.front().c;
    if (!small.empty()) C.max_c[1] = small.front().c;
    C.blocks.insert(C.blocks.end(), small.begin(), small.end());
    return C;
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
    const int c = std::max(C.max_c[0], C.max_c[1]);
    if (c > 0) {
        int tr = 16;
        auto bytes = [&](int t) { return sizeof(double) * ((size_t)t * c + (size_t)t * kInvWarps + (size_t)kInvWarps * c); };
        while (tr > 1 && bytes(tr) > room) tr /= 2;
        MSP_CUDA(cudaFuncSetAttribute(patch_inverse_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes(tr)));
        for (size_t b0 = 0; b0 < C.blocks.size(); b0 += 65535) {
            const unsigned nb = (unsigned)std::min<size_t>(65535, C.blocks.size() - b0);
            patch_inverse_kernel<<<dim3((c + kInvWarps - 1) / kInvWarps, nb), 32 * kInvWarps, bytes(tr), s>>>(
                blocks + b0, L, F, Fi, status, tr);
            count_launches(1);
        }
        MSP_CUDA(cudaGetLastError());
    }
    return MSP_OK;
}

}  // namespace msp
