// Device-side state of the ADMM / L-BFGS solver: every vector lives in the
// panel layout of the stacked unknown (2 * n floats), every scalar decision
// (step length, pair acceptance, memory reset) stays in device memory so the
// whole solve is a fixed sequence of launches with no host round trip.
#pragma once

#include "internal.h"

namespace tlr {

enum ScalarSlot { SC_ALPHA = 0, SC_F, SC_F0, SC_C0, SC_C1, SC_C2, SC_C3, SC_C4, SC_GAMMA, SC_COUNT };
// SI_RFLAG: 1 when this iteration's direction failed the descent test and was
// replaced by -g (the iteration already counts as a restart)
enum IntSlot { SI_CNT = 0, SI_NEWEST, SI_ITERS, SI_RESTARTS, SI_STATUS, SI_RFLAG, SI_COUNT };

// after the counters: [SI_COUNT + 1] the contractions' error word, then the block
// counters of the passes whose last block finishes their sums (zero between launches)
enum CounterSlot { CT_LINE = SI_COUNT + 2, CT_PAIR, CT_DIR };   // CT_DIR: 1 + kLbClusters of them

// compact L-BFGS: pairs per inner-product pass; a block leaves kLbVals partials (a
// row of kLbRow), the last block of every kLbCluster adds its cluster's up
constexpr int kLbGroup = 10, kLbGroups = (32 + kLbGroup - 1) / kLbGroup;
constexpr int kLbVals = 5 * kLbGroup + 1, kLbRow = kLbVals + 1;
constexpr int kLbCluster = 16, kLbClusters = (kRedBlocks + kLbCluster - 1) / kLbCluster;
constexpr long long kLbSumOff = (long long)kLbGroups * kRedBlocks * kLbRow;
constexpr long long kLbPartDoubles = kLbSumOff + (long long)kLbGroups * kLbClusters * kLbRow;

struct SolverDev {
    long long n2;        // floats per theta-space vector (2 * n_theta)
    int m;               // L-BFGS memory
    int ring;            // m + 1 slots: the slot after the newest is always free
    float *x, *z, *u, *v, *g, *gf, *d;
    float *sh, *yh;      // ring of s and y vectors, ring * n2 floats each
    double* acoef;       // [64] direction coefficients: [j] of s_j, [32 + j] of y_j (j-th newest)
    double* SYm;         // [ring * ring] <s_a, y_b> by slot
    double* YYm;         // [ring * ring] <y_a, y_b> by slot
    double* lbpart;      // partials of the direction's inner products ...
    double* lbsum;       // ... and their cluster sums
    unsigned* lbctr;     // block counters: [0] clusters, [1 + i] blocks of cluster i (zero between launches)
    double* sc;          // ScalarSlot values
    int* ints;           // IntSlot values
    double* fhist;       // [TLR_MAX_HIST]
    double* part3;       // 3 * kRedBlocks: <x-v,x-v>, <x-v,d>, <d,d> partials of the direction pass
    double* part6;       // 6 * kRedBlocks: line-search inner products
    double* partp;       // 3 * kRedBlocks: the new pair's inner products
};

// blocks of a reduction over n values: enough work for 256 threads each, at most
// kRedBlocks (a function of n alone, so the order of every sum is fixed)
inline int red_blocks(long long n) {
    const long long b = (n + 1023) / 1024;
    return (int)(b < 1 ? 1 : b > kRedBlocks ? kRedBlocks : b);
}

// partials of ||R||^2 (n complex) into part[red_blocks(n)]
cudaError_t sv_norm_part(const cf* R, long long n, double* part, cudaStream_t st);
// f0 = f = 0.5 sum of the np partials
cudaError_t sv_record_f0(const SolverDev& S, const double* partf, long long np, cudaStream_t st);
cudaError_t sv_admm_init(const SolverDev& S, cudaStream_t st);
cudaError_t sv_admm_resume(const SolverDev& S, cudaStream_t st);
cudaError_t sv_xupdate_start(const SolverDev& S, double rho, cudaStream_t st);
// the direction d, and the partials of the theta-space line-search products
cudaError_t sv_direction(const SolverDev& S, cudaStream_t st);
// The line search: the six inner products of Rf, A1, A2 (n complex, FP32), or with
// Rf read from its KN packing (kn[i], as rstep writes it, over rstep's tiles), then
// phi's minimiser by the last block.
cudaError_t sv_line_search(const SolverDev& S, const cf* R, const cf* A1, const cf* A2, long long n, double rho,
                           cudaStream_t st);
cudaError_t sv_line_search_packed(const SolverDev& S, char* const* kn, const cf* A1, const cf* A2, int nr, int ns, int b,
                                  const long long* roff, int nblk, int fmt, double rho, cudaStream_t st);
// R += a A1 + a^2 A2 (a = *alpha) with partials of ||R||^2 into partf[red_blocks(n)]
cudaError_t sv_step_residual(cf* R, const cf* A1, const cf* A2, long long n, const double* alpha,
                             double* partf, cudaStream_t st);
cudaError_t sv_step_theta(const SolverDev& S, cudaStream_t st);
// The gradient's split-K partials summed into gf (as reduce_grad does), the new
// pair (s, y) and g from it, and, by the last block, f from the nf residual-norm
// partials and the acceptance of the pair.
cudaError_t sv_gradient_pair(const SolverDev& S, const cf* part, int nsplit, long long nlr, long long ndense,
                             long long b, int general, const long long* zoff, const int* zdim, double rho,
                             const double* partf, long long nf, cudaStream_t st);
cudaError_t sv_admm_zu(const SolverDev& S, double lam, double rho, cudaStream_t st);

}  // namespace tlr
