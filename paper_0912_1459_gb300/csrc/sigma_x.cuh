// FP64 self-energy from exact-slice tensor-core integrals (sigma_x.cu).
#pragma once

#include "sigma.cuh"

namespace cds {

// Bases this large take the tensor-core integrals and the evaluation kernels
// of sigma_x.cu; smaller ones the fused FP64 kernel (k_sigma_fp64).  The
// cached Newton passes follow the same rule, so both read one arithmetic.
bool sigma_x_serves(int32_t nmo, int32_t nocc, int32_t np);
// The workspace to ask for (at most 4 GB; 0: none that small serves), and whether one of
// ws_bytes serves: below everything at once the spectators are taken in panels.
size_t sigma_x_bytes(int32_t nmo, int32_t nocc, int32_t M, int32_t np, int32_t nE);
bool sigma_x_fits(int32_t nmo, int32_t nocc, int32_t M, int32_t np, int32_t nE, size_t ws_bytes);
// sigma / dsigma [np][nE]; cache (may be null): receives the numerators in the
// item layout of k_sigma_fp64.  resplit = false keeps the operands (and, where
// every orbital's integrals fit the workspace at once, the integrals) of the
// previous call with the same factors and workspace.
int sigma2_x(int32_t nmo, int32_t nocc, int32_t M, const double* Lov, const double* Lp, int32_t np,
             const double* eps, const double* E, int32_t nE, const int32_t* active, double* sigma,
             double* dsigma, void* ws, size_t ws_bytes, cudaStream_t stream, bool resplit, double* cache);
// One energy per orbital (E [np]) from stored numerators; part: two doubles per item.
int sigma2_x_cached(int32_t nmo, int32_t nocc, int32_t np, const double* eps, const double* E,
                    const int32_t* active, const double* cache, double* sigma, double* dsigma,
                    double* part, cudaStream_t stream);
// Eq. MP2: e_pair[nocc].
size_t mp2_x_bytes(int32_t nmo, int32_t nocc, int32_t M);
bool mp2_x_fits(int32_t nmo, int32_t nocc, int32_t M, size_t ws_bytes);
int mp2_x(int32_t nmo, int32_t nocc, int32_t M, const double* Lov, const double* eps,
          double* e_pair, void* ws, size_t ws_bytes, cudaStream_t stream);

}  // namespace cds
