// Dense factorisations of the patches' small symmetric and square blocks on
// thread-block clusters: one patch on one CTA, or on eight when it would otherwise
// keep a single SM busy after the others have finished.
#pragma once
#include "internal.h"

namespace msp {

// One patch's c x c block (column-major, leading dimension c) in the stacked arrays.
struct PatchBlock {
    long long off;
    int c;
    int idx;      // patch
};

constexpr int kPatchCluster = 8;   // CTAs of a patch that takes a cluster (the portable limit)

// Patches that take a cluster each, then those that take one CTA, both largest first.
struct PatchClasses {
    std::vector<PatchBlock> blocks;
    int n_big = 0;
    int max_c[2] = {0, 0};         // largest order of either class
};
PatchClasses classify_patches(const std::vector<int>& cols, const std::vector<long long>& off);

// Cholesky of every block G (lower triangle read) + shift I, shift = shift_scale[patch]
// trace(G) (shifted != 0; else 0), on a non-positive pivot a growing shift (1e-14 trace
// if it was zero, else x 100), at most six tries: status[patch] = tries, or -1.
// F = L^T and Fi = L^{-T}; L is overwritten.  `blocks` is C.blocks on the device.
msp_status patch_cholesky(const PatchClasses& C, const PatchBlock* blocks, const double* G, double* L, double* F,
                          double* Fi, const double* shift_scale, bool shifted, int* status, cudaStream_t s);

// Fi = L^{-T} of every lower triangular block
msp_status patch_triangular_inverse(const PatchClasses& C, const PatchBlock* blocks, const double* L, double* Fi,
                                    cudaStream_t s);

// Householder QR with column pivoting T P = Q R of every block: W = R^T and Q, the
// preconditioner of the Jacobi sweeps in the manner of Drmac and Veselic (2008): the
// sweeps run on the columns of R^T, whose rows decay with the pivots, with V started at Q,
// so that their rotations J leave V = Q J, the left singular vectors of T (the
// permutation only acts on the right).  R and cols are work blocks as large as T.  On
// clusters, or one CTA per patch where the patches keep all SMs busy.
msp_status patch_qrcp(const PatchClasses& C, const PatchBlock* blocks, const double* T, double* W, double* Q, double* R,
                      double* cols, cudaStream_t s);

// FP64 one-sided Jacobi sweeps of every block (W rotated to U S, V accumulating) with
// each patch on a cluster; `all` largest first.  Returned in `rest`, for the sweeps on one CTA
// each: the blocks whose columns a cluster's shared memory does not hold, or all of them where
// that ends sooner.  d_blocks is read until the stream has passed the launches.
msp_status patch_jacobi(const std::vector<PatchBlock>& all, double* W, double* V, int max_sweeps, double tol,
                        double small_rel, int* sweeps, DevBuf<PatchBlock>& d_blocks, std::vector<PatchBlock>& rest,
                        cudaStream_t s);

}  // namespace msp
