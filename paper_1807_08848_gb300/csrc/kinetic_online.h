// Online stage of the kinetic slab (kinetic_online.cu).
#pragma once
#include "kinetic_internal.h"

namespace msp {

struct KOnArgs {
    int M, nv, N, k_max;
    const double* v;
    const KPatchDev* patches;
    const int* k;
    const int* c_off;
    const long long* q_off;
    const double* Q;
    const long long* l_off;      // k_m x k_m blocks: L_m, L_m^{-T}
    const long long* cb_off;     // k_{m+1} x k_m blocks: C_m and the chains' matrices
    const double* Fi;            // L_m^{-T}
    const double* Tf;            // L_{m+1}^{-1} C_m (k_{m+1} x k_m)
    const double* Tb;            // L_m^{-T} C_m^T (k_m x k_{m+1})
};

// The factor and the matrices of the chains (host tables k, l_off, cb_off); *failed = 1 on a
// non-positive pivot.  Synchronises.
msp_status kinetic_factor(const KOnArgs& A, const std::vector<int>& k, const std::vector<long long>& l_off,
                          const std::vector<long long>& cb_off, double* Lf, double* Cf, double* Fi, double* Tf, double* Tb,
                          int* failed, cudaStream_t s);

// c = argmin |P c - d| per data set and its field.  Synchronises.
msp_status kinetic_online(const KOnArgs& A, int Np, const double* inflow, int batch, double* f_out, double* c_out,
                          cudaStream_t s);

}  // namespace msp
