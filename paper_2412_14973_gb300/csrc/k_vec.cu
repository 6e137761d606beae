// theta-space and reduction kernels: the layout maps between the stacked
// unknown (Z-bar, L-bar, R-bar) and the block panels, the gradient split-K
// reduction with the dense-tile symmetrisation (eq. 26), FP64 inner products,
// the exact line search on the quartic phi(alpha), and the L-BFGS direction
// (compact form) / ADMM updates (eq. 19-24) with every scalar kept on the device.
//
// All reductions run on a grid that depends on the length alone (red_blocks) and
// sum their per-block partials in a fixed order, so results are bitwise
// reproducible.  An iteration of a small solve is a chain of launches, so the
// passes are few and finish their own sums: the last block to arrive adds the
// partials up and makes the scalar decision (direction coefficients, step length,
// pair acceptance), where each was a launch of its own with one block.
#include <algorithm>

#include "internal.h"
#include "pack.h"
#include "reduce.h"
#include "solver_dev.h"

namespace tlr {

// ---------------------------------------------------------------------------
// helpers
// ---------------------------------------------------------------------------
// Sum of n partials by a block of 256 threads in a fixed order, in every thread;
// four independent sums per thread keep the loads in flight.
__device__ __forceinline__ double sum_part(const double* part, long long n, double (*sh)[256]) {
    double a0 = 0.0, a1 = 0.0, a2 = 0.0, a3 = 0.0;
    long long i = threadIdx.x;
    for (; i + 768 < n; i += 1024) {
        a0 += part[i];
        a1 += part[i + 256];
        a2 += part[i + 512];
        a3 += part[i + 768];
    }
    for (; i < n; i += 256) a0 += part[i];
    const double v[1] = {(a0 + a1) + (a2 + a3)};
    (void)block_sums(v, sh);
    const double r = sh[0][0];
    __syncthreads();
    return r;
}

// Sums of K interleaved partial slabs (part[i K + k], i < n) by a block of 256
// threads: one warp per sum, lanes over i.  Thread k < K returns sum k.
template <int K>
__device__ __forceinline__ double sum_slabs(const double* part, int n, double* sh) {
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    if (w < K) {
        double a0 = 0.0, a1 = 0.0;
        int i = l;
        for (; i + 32 < n; i += 64) {
            a0 += part[i * K + w];
            a1 += part[(i + 32) * K + w];
        }
        if (i < n) a0 += part[i * K + w];
        const double r = warp_sum(a0 + a1);
        if (l == 0) sh[w] = r;
    }
    __syncthreads();
    const double r = threadIdx.x < K ? sh[threadIdx.x] : 0.0;
    __syncthreads();
    return r;
}

#define GRID_STRIDE(i, n) \
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < (n); i += (long long)gridDim.x * blockDim.x)

// ---------------------------------------------------------------------------
// layout maps
// ---------------------------------------------------------------------------
// Row a of panel column g, one block row of threads over 32 columns and 8 rows
// (the columns' maps are read once per thread and 64 rows; a grid-stride loop with
// a 64-bit division and a map lookup per value took 64 us for 64 MB).
template <bool TO_PANEL>
__global__ void __launch_bounds__(256) k_panel_map(PanelMap m, const cf* __restrict__ src, cf* __restrict__ dst,
                                                   int gcols, int grows) {
    chain_entry();
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    const long long nlb = (long long)gcols * grows;
    for (long long e = blockIdx.x; e < nlb; e += gridDim.x) {
        const long long g = e % gcols * 32 + tx;
        const int a0 = (int)(e / gcols) * 64 + ty;
        if (g >= m.Ktot) continue;
        const int rows = min(m.colrows[g], a0 - ty + 64);
        const long long tb = m.colsrc[g], pb = m.colpan[g];
        const int ts = m.colstride[g], ps = m.panstride[g];
#pragma unroll 8
        for (int a = a0; a < rows; a += 8) {
            const long long t = tb + (long long)a * ts, p = pb + (long long)a * ps;
            if (TO_PANEL)
                dst[p] = src[t];
            else
                dst[t] = src[p];
        }
    }
    const long long bb = m.b * m.b;
    GRID_STRIDE(e, m.ndense * bb) {
        const long long t = e / bb, r = (e % bb) / m.b, c = e % m.b, n = m.zdim[t];
        if (r < n && c < n) {
            const long long th = m.zsrc[t] + r * n + c, pa = m.zbase + m.zoff[t] + r * n + c;
            if (TO_PANEL)
                dst[pa] = src[th];
            else
                dst[th] = src[pa];
        }
    }
}

static cudaError_t panel_map(const PanelMap& m, bool to_panel, const cf* src, cf* dst, cudaStream_t st) {
    const long long gc = (m.Ktot + 31) / 32, gr = (m.b + 63) / 64;
    const long long want = std::max(gc * gr, (m.ndense * m.b * m.b + 1023) / 1024);
    const unsigned grid = (unsigned)std::max(1LL, std::min(want, 152LL * 64));
    if (to_panel)
        (void)launch_pass(k_panel_map<true>, dim3(grid), dim3(256), st, m, src, dst, (int)gc, (int)gr);
    else
        (void)launch_pass(k_panel_map<false>, dim3(grid), dim3(256), st, m, src, dst, (int)gc, (int)gr);
    counted(1);
    return cudaGetLastError();
}

cudaError_t theta_to_panel(const PanelMap& m, const cf* theta, cf* pan, cudaStream_t st) {
    return panel_map(m, true, theta, pan, st);
}
cudaError_t panel_to_theta(const PanelMap& m, const cf* pan, cf* theta, cudaStream_t st) {
    return panel_map(m, false, pan, theta, st);
}

// Dense tile t of a panel-ordered region: (offset, size) from the per-tile
// tables, or the t-th of equal tiles of size b.
__device__ __forceinline__ bool dense_tile(long long e, long long b, const long long* zoff, const int* zdim,
                                           long long& base, long long& n, long long& r, long long& c) {
    const long long bb = b * b;
    long long t;
    if (e < 0x7fffffffLL && bb < 0x7fffffffLL) {   // 64-bit divisions are long sequences
        const unsigned ue = (unsigned)e, ub = (unsigned)b, ubb = (unsigned)bb, ut = ue / ubb, q = ue - ut * ubb;
        t = ut;
        r = q / ub;
        c = q - (unsigned)r * ub;
    } else {
        t = e / bb;
        r = (e % bb) / b;
        c = e % b;
    }
    if (!zoff) {
        base = t * bb;
        n = b;
        return true;
    }
    base = zoff[t];
    n = zdim[t];
    return r < n && c < n;
}

// Zs = (Z + Z^T)/2 (reciprocal form: the symmetrisation preconditioner P of
// eq. 7, X_ii = P Z_ii) or Z^T (general form: row block i of Y = X^T Dfrak
// takes X_ii^T)
__global__ void k_sym_dense(const cf* __restrict__ pan, long long zbase, long long ndense, long long b,
                            cf* __restrict__ Zs, int general, const long long* __restrict__ zoff,
                            const int* __restrict__ zdim) {
    chain_entry();
    GRID_STRIDE(e, ndense * b * b) {
        long long base, n, r, c;
        if (!dense_tile(e, b, zoff, zdim, base, n, r, c)) continue;
        const cf u = pan[zbase + base + r * n + c];
        const cf v = pan[zbase + base + c * n + r];
        Zs[base + r * n + c] = general ? v : make_float2(0.5f * (u.x + v.x), 0.5f * (u.y + v.y));
    }
}

cudaError_t sym_dense(const cf* pan, long long zbase, long long ndense, long long b, cf* Zs, cudaStream_t st,
                      int general, const long long* zoff, const int* zdim) {
    if (ndense == 0) return cudaSuccess;
    (void)launch_pass(k_sym_dense, dim3(512), dim3(256), st, pan, zbase, ndense, b, Zs, general, zoff, zdim);
    counted(1);
    return cudaGetLastError();
}

// one gradient entry: its split-K partials (compensated, fixed order) ...
__device__ __forceinline__ cf split_sum(const cf* __restrict__ part, int nsplit, long long stride, long long e) {
    Acc x, y;
#pragma unroll 4
    for (int c = 0; c < nsplit; ++c) {
        const cf v = part[c * stride + e];
        x.add(v.x);
        y.add(v.y);
    }
    return make_float2((float)x.val(), (float)y.val());
}
// ... of a dense tile: (G + G^T)/2 (reciprocal form) or G^T (general form); e1 the
// entry, e2 its mirror
__device__ __forceinline__ cf split_sum_dense(const cf* __restrict__ part, int nsplit, long long stride, long long e1,
                                              long long e2, int general) {
    Acc x, y;
    for (int c = 0; c < nsplit; ++c) {
        const cf v = part[c * stride + e2];
        if (!general) {
            const cf u = part[c * stride + e1];
            x.add(u.x);
            y.add(u.y);
        }
        x.add(v.x);
        y.add(v.y);
    }
    const double s = general ? 1.0 : 0.5;
    return make_float2((float)(s * x.val()), (float)(s * y.val()));
}

// grad = sum of split-K partials
__global__ void k_reduce_grad(const cf* __restrict__ part, int nsplit, long long stride, long long nlr,
                              long long ndense, long long b, cf* __restrict__ grad, int general,
                              const long long* __restrict__ zoff, const int* __restrict__ zdim) {
    chain_entry();
    GRID_STRIDE(e, nlr) grad[e] = split_sum(part, nsplit, stride, e);
    GRID_STRIDE(e, ndense * b * b) {
        long long base, n, r, q;
        if (!dense_tile(e, b, zoff, zdim, base, n, r, q)) continue;
        const long long e1 = nlr + base + r * n + q, e2 = nlr + base + q * n + r;
        grad[e1] = split_sum_dense(part, nsplit, stride, e1, e2, general);
    }
}

cudaError_t reduce_grad(const cf* part, int nsplit, long long stride, long long nlr, long long ndense,
                        long long b, cf* grad, cudaStream_t st, int general, const long long* zoff,
                        const int* zdim) {
    (void)launch_pass(k_reduce_grad, dim3(1024), dim3(256), st, part, nsplit, stride, nlr, ndense, b, grad, general,
                      zoff, zdim);
    counted(1);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// FP64 inner products
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_sum_partials(const double* part, long long n, double scale, double* out) {
    chain_entry();
    __shared__ double sh[1][256];
    const double v = sum_part(part, n, sh);
    if (threadIdx.x == 0) out[0] = scale * v;
}

cudaError_t sum_partials(const double* part, long long n, double scale, double* out, cudaStream_t st) {
    (void)launch_pass(k_sum_partials, dim3(1), dim3(256), st, part, n, scale, out);
    counted(1);
    return cudaGetLastError();
}

// Re<R,R>, Re<R,A1>, Re<R,A2>, Re<A1,A1>, Re<A1,A2>, Re<A2,A2>
__device__ __forceinline__ void dots6_add(Acc* s, float rx, float ry, float ax, float ay, float cx, float cy) {
    s[0].add(fmaf(rx, rx, ry * ry));
    s[1].add(fmaf(rx, ax, ry * ay));
    s[2].add(fmaf(rx, cx, ry * cy));
    s[3].add(fmaf(ax, ax, ay * ay));
    s[4].add(fmaf(ax, cx, ay * cy));
    s[5].add(fmaf(cx, cx, cy * cy));
}

// the six products of one complex element added to t (plain FP32: a group of
// up to four elements is summed like this before one compensated add, so
// the group's rounding is of the order of the products' own)
__device__ __forceinline__ void dots6_group(float* t, float rx, float ry, float ax, float ay, float cx, float cy) {
    t[0] += fmaf(rx, rx, ry * ry);
    t[1] += fmaf(rx, ax, ry * ay);
    t[2] += fmaf(rx, cx, ry * cy);
    t[3] += fmaf(ax, ax, ay * ay);
    t[4] += fmaf(ax, cx, ay * cy);
    t[5] += fmaf(cx, cx, cy * cy);
}

// R += a A1 + a^2 A2 ; partial of ||R_new||^2 -> part[blk]
__global__ void __launch_bounds__(kRedThreads) k_step_residual(cf* __restrict__ R, const cf* __restrict__ A1,
                                                              const cf* __restrict__ A2, long long n,
                                                              const double* __restrict__ alpha, double* part) {
    chain_entry();
    __shared__ double sh[1][256];
    const float a = (float)alpha[0];
    const float a2 = (float)(alpha[0] * alpha[0]);
    Acc s;
    GRID_STRIDE(i, n) {
        cf r = R[i];
        if (a != 0.f) {
            const cf u = A1[i], w = A2[i];
            r.x = fmaf(a2, w.x, fmaf(a, u.x, r.x));
            r.y = fmaf(a2, w.y, fmaf(a, u.y, r.y));
            R[i] = r;
        }
        s.add(fmaf(r.x, r.x, r.y * r.y));
    }
    const double v[1] = {s.val()};
    const double t = block_sums(v, sh);
    if (threadIdx.x == 0) part[blockIdx.x] = t;
}

__global__ void k_axpy_dev(float* __restrict__ x, const float* __restrict__ y, long long n2,
                           const double* __restrict__ alpha) {
    chain_entry();
    const float a = (float)alpha[0];
    if (a == 0.f) return;
    GRID_STRIDE(i, n2) x[i] = fmaf(a, y[i], x[i]);
}

cudaError_t axpy_dev(float* x, const float* y, long long n2, const double* alpha, cudaStream_t st) {
    (void)launch_pass(k_axpy_dev, dim3(1024), dim3(256), st, x, y, n2, alpha);
    counted(1);
    return cudaGetLastError();
}

// ===========================================================================
// Solver kernels (L-BFGS two-loop recursion, exact line search, ADMM).
// ===========================================================================

// partials of ||R||^2
__global__ void __launch_bounds__(kRedThreads) k_norm_part(const cf* __restrict__ R, long long n, double* part) {
    chain_entry();
    __shared__ double sh[1][256];
    Acc s;
    GRID_STRIDE(i, n) {
        const cf r = R[i];
        s.add(fmaf(r.x, r.x, r.y * r.y));
    }
    const double v[1] = {s.val()};
    const double t = block_sums(v, sh);
    if (threadIdx.x == 0) part[blockIdx.x] = t;
}

// g = gf + rho (x - v); history cleared (start of an x-update)
__global__ void k_xupdate_start(SolverDev S, double rho) {
    chain_entry();
    const float r = (float)rho;
    GRID_STRIDE(i, S.n2) S.g[i] = S.gf[i] + r * (S.x[i] - S.v[i]);
    if (blockIdx.x == 0 && threadIdx.x == 0) S.ints[SI_CNT] = 0;
}

__device__ __forceinline__ int ring_idx(const SolverDev& S, int j) {
    // j-th newest pair (0 = newest)
    const int R = S.ring;
    return ((S.ints[SI_NEWEST] - j) % R + R) % R;
}

// L-BFGS direction d = -H g in the compact form of the inverse BFGS update
// (Byrd, Nocedal and Schnabel 1994): with the k stored pairs ordered oldest
// first, S = [s_1 .. s_k], Y = [y_1 .. y_k], R = triu(S^T Y), D = diag(S^T Y),
// H0 = gamma I and gamma = <s,y>/<y,y> of the newest pair,
//   H g = gamma g + S a - gamma Y u,  u = R^-1 S^T g,
//   a = R^-T ((D + gamma Y^T Y) u - gamma Y^T g).
// This is the matrix the two-loop recursion applies, evaluated in three
// steps: the inner products (passes over groups of pairs; they also fill the
// newest pair's row and column of S^T Y and Y^T Y, which are kept by slot),
// the small FP64 triangular solves in one block, and one combination pass.

// partials per block: for pair j of the group, <s_j,g>, <y_j,g>, <s_j,y_n>,
// <s_n,y_j>, <y_j,y_n> (n = the newest pair).  Per-thread sums are plain FP32
// multiply-adds (one term per 77824 values: a few dozen at the large sizes), combined
// in FP64 across threads and blocks: these products only set the direction's
// coefficients, whose rounding the exact line search and the descent test absorb.
// 128 threads of <= 128 registers: a CTA fits beside the two GEMM CTAs of an SM
constexpr int kLbThreads = 128;
constexpr int kLbLd = kLbThreads + 8;   // row length of the block's sums: 4 rows read together lie in different banks

__device__ void lb_solve(const SolverDev& S, int cnt, int ncl, double* val, double* mat);

// Blocks of the direction's inner products: one value of each vector per thread until
// there are kRedBlocks, so that up to 77824 values every product goes to the FP64 sums
// by itself
inline int lb_blocks(long long n2) {
    const long long b = (n2 + kLbThreads - 1) / kLbThreads;
    return (int)(b < 1 ? 1 : b > kRedBlocks ? kRedBlocks : b);
}

// last != 0: the launch over the last group of pairs, whose last block finishes
// the direction's coefficients (lb_solve).  FP64 adds and conversions run at 2 lanes
// per cycle on this part, so a lane adds its 16 terms of a value up as an exact FP32
// sum with its errors (Acc2: no fewer bits than FP64) and 8 lanes meet in FP64.  With
// FP64 adds throughout, a solve of 256 receivers took 3.64 ms (3.37 here).
__global__ void __launch_bounds__(kLbThreads, 4) k_lb_dots(SolverDev S, int j0, int last) {
    chain_entry();
    __shared__ __align__(16) float shv[kLbVals * kLbLd];
    const int cnt = S.ints[SI_CNT];
    if (j0 < cnt) {
        const int jc = min(kLbGroup, cnt - j0);
        const float* sp[kLbGroup];
        const float* yp[kLbGroup];
#pragma unroll
        for (int jj = 0; jj < kLbGroup; ++jj) {
            const int idx = ring_idx(S, jj < jc ? j0 + jj : j0);
            sp[jj] = S.sh + (long long)idx * S.n2;
            yp[jj] = S.yh + (long long)idx * S.n2;
        }
        const int nw = ring_idx(S, 0);
        const float* sn = S.sh + (long long)nw * S.n2;
        const float* yn = S.yh + (long long)nw * S.n2;
        float acc[kLbGroup][5];
#pragma unroll
        for (int jj = 0; jj < kLbGroup; ++jj)
#pragma unroll
            for (int t = 0; t < 5; ++t) acc[jj][t] = 0.f;
        float gg = 0.f;   // <g, g> for the descent test (first group only)
        GRID_STRIDE(i, S.n2) {
            const float gi = S.g[i], sni = sn[i], yni = yn[i];
            gg = fmaf(gi, gi, gg);
#pragma unroll
            for (int jj = 0; jj < kLbGroup; ++jj) {
                if (jj < jc) {
                    const float s = sp[jj][i], y = yp[jj][i];
                    acc[jj][0] = fmaf(s, gi, acc[jj][0]);
                    acc[jj][1] = fmaf(y, gi, acc[jj][1]);
                    acc[jj][2] = fmaf(s, yni, acc[jj][2]);
                    acc[jj][3] = fmaf(sni, y, acc[jj][3]);
                    acc[jj][4] = fmaf(y, yni, acc[jj][4]);
                }
            }
        }
#pragma unroll
        for (int jj = 0; jj < kLbGroup; ++jj)
#pragma unroll
            for (int t = 0; t < 5; ++t) shv[(jj * 5 + t) * kLbLd + threadIdx.x] = acc[jj][t];
        shv[5 * kLbGroup * kLbLd + threadIdx.x] = gg;
        __syncthreads();
        const int l8 = threadIdx.x & 7;
        double* const mine = S.lbpart + ((long long)(j0 / kLbGroup) * kRedBlocks + blockIdx.x) * kLbRow;
        for (int v0 = 0; v0 < kLbVals; v0 += kLbThreads / 8) {
            const int v = v0 + (threadIdx.x >> 3);   // 8 lanes per value
            const float* row = shv + min(v, kLbVals - 1) * kLbLd;
            Acc2 a;
#pragma unroll
            for (int i = 0; i < kLbThreads / 8; ++i) a.add(row[l8 + 8 * i]);
            double r = a.val();
            if (!isfinite(r)) {   // Inf, NaN or sums beyond FP32
                r = 0.0;
                for (int i = 0; i < kLbThreads / 8; ++i) r += (double)row[l8 + 8 * i];
            }
#pragma unroll
            for (int o = 4; o > 0; o >>= 1) r += __shfl_down_sync(0xffffffffu, r, o, 8);
            if (l8 == 0 && v < kLbVals) mine[v] = r;
        }
    }
    // The last block of every 16 adds its cluster's partials up, the last of those
    // finishes: a thread per value, and 16 (38) additions each on as many SMs, where
    // one block adding 608 x 51 doubles took 10 us.
    const int cl = blockIdx.x / kLbCluster, ncl = (gridDim.x + kLbCluster - 1) / kLbCluster;
    const int in_cl = min(kLbCluster, (int)gridDim.x - cl * kLbCluster);
    unsigned* const ctr = reinterpret_cast<unsigned*>(S.lbctr);
    if (!last_block(ctr + 1 + cl, in_cl)) return;
    const int grp = j0 / kLbGroup, t = threadIdx.x;
    if (j0 < cnt && t < kLbVals) {
        const double* q = S.lbpart + ((long long)grp * kRedBlocks + cl * kLbCluster) * kLbRow + t;
        double a = 0.0;
#pragma unroll 4
        for (int i = 0; i < in_cl; ++i) a += q[(long long)i * kLbRow];
        S.lbsum[((long long)grp * kLbClusters + cl) * kLbRow + t] = a;
    }
    if (!last || !last_block(ctr, ncl)) return;
    double* const mat = reinterpret_cast<double*>(shv);   // 2 x 32 x 33 doubles and 161 values
    lb_solve(S, cnt, ncl, mat + 2 * 32 * 33, mat);
}
static_assert(sizeof(double) * (2 * 32 * 33 + 161) <= sizeof(float) * kLbVals * kLbLd, "lb_solve's storage");

// One block: finalise the cluster sums (a thread per value, fixed order), update the
// newest pair's row / column of S^T Y and Y^T Y, then (warp 0, a lane per
// pair) the triangular solves; coefficients to acoef, gamma to sc[SC_GAMMA].
__device__ void lb_solve(const SolverDev& S, int cnt, int ncl, double* val, double* mat) {
    double* const Rm = mat;
    double* const Ym = mat + 32 * 33;
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    if (cnt == 0) {
        // d = -g, a descent direction unless g = 0 (which the line search meets)
        if (threadIdx.x == 0) {
            S.ints[SI_RFLAG] = 0;
            S.sc[SC_GAMMA] = 1.0;
        }
        return;
    }
    const int R = S.ring, k = cnt;
    const int nw = ring_idx(S, 0);
    // val[5 j + kind] of the j-th newest pair, val[5 cnt] = <g, g>
    for (int v = threadIdx.x; v <= 5 * cnt; v += kLbThreads) {
        const int grp = v == 5 * cnt ? 0 : v / (5 * kLbGroup), t = v == 5 * cnt ? kLbVals - 1 : v % (5 * kLbGroup);
        const double* q = S.lbsum + (long long)grp * kLbClusters * kLbRow + t;
        double a0 = 0.0, a1 = 0.0;
#pragma unroll 4
        for (int i = 0; i + 1 < ncl; i += 2) {
            a0 += q[(long long)i * kLbRow];
            a1 += q[(long long)(i + 1) * kLbRow];
        }
        if (ncl & 1) a0 += q[(long long)(ncl - 1) * kLbRow];
        val[v] = a0 + a1;
    }
    // oldest first: position i holds the (cnt - 1 - i)-th newest pair; the newest
    // pair's row and column come from val below
    for (int e = threadIdx.x; e < k * k; e += kLbThreads) {
        const int i = e / k, j = e - i * k;
        const int si = ring_idx(S, k - 1 - i), sj = ring_idx(S, k - 1 - j);
        if (si != nw && sj != nw) {
            Rm[i * 33 + j] = S.SYm[si * R + sj];
            Ym[i * 33 + j] = S.YYm[si * R + sj];
        }
    }
    __syncthreads();
    if (threadIdx.x < cnt) {
        const int j = threadIdx.x, a = ring_idx(S, j), i = k - 1 - j;
        const double sy = val[j * 5 + 2], ys = val[j * 5 + 3], yy = val[j * 5 + 4];   // <s_j,y_n>, <s_n,y_j>, <y_j,y_n>
        S.SYm[a * R + nw] = sy;
        if (j > 0) S.SYm[nw * R + a] = ys;
        S.YYm[a * R + nw] = yy;
        S.YYm[nw * R + a] = yy;
        Rm[i * 33 + k - 1] = sy;
        if (j > 0) Rm[(k - 1) * 33 + i] = ys;
        Ym[i * 33 + k - 1] = yy;
        Ym[(k - 1) * 33 + i] = yy;
    }
    __syncthreads();
    if (w != 0) return;
    // lane i holds position i
    const bool on = l < k;
    const double p = on ? val[(k - 1 - l) * 5] : 0.0, q = on ? val[(k - 1 - l) * 5 + 1] : 0.0;
    const double dia = on ? Rm[l * 33 + l] : 1.0, inv = 1.0 / dia;
    const double gamma = Rm[(k - 1) * 33 + (k - 1)] / Ym[(k - 1) * 33 + (k - 1)];
    // u = R^-1 p (R upper triangular)
    double u = p;
    for (int i = k - 1; i >= 0; --i) {
        const double ui = __shfl_sync(0xffffffffu, u * inv, i);
        if (l == i) u = ui;
        if (l < i) u -= Rm[l * 33 + i] * ui;
    }
    // t = D u + gamma Y^T Y u - gamma q
    double t = dia * u - gamma * q;
    for (int j = 0; j < k; ++j) {
        const double uj = __shfl_sync(0xffffffffu, u, j);
        if (on) t += gamma * Ym[l * 33 + j] * uj;
    }
    // a = R^-T t (R^T lower triangular)
    for (int i = 0; i < k; ++i) {
        const double ai = __shfl_sync(0xffffffffu, t * inv, i);
        if (l == i) t = ai;
        if (on && l > i) t -= Rm[i * 33 + l] * ai;
    }
    // descent test: <g, d> = -(gamma <g,g> + sum_i a_i <s_i,g> - gamma sum_i u_i <y_i,g>)
    double gd = warp_sum(on ? t * p - gamma * u * q : 0.0);
    gd = -(gamma * val[5 * k] + __shfl_sync(0xffffffffu, gd, 0));
    if (!(gd < 0.0)) {
        // not a descent direction: clear the memory and take d = -g in this
        // same iteration (the restart of L-BFGS)
        if (l == 0) {
            S.ints[SI_CNT] = 0;
            S.ints[SI_RESTARTS] += 1;
            S.ints[SI_RFLAG] = 1;
            S.sc[SC_GAMMA] = 1.0;
        }
        return;
    }
    if (on) {
        S.acoef[k - 1 - l] = t;   // j-th newest
        S.acoef[32 + k - 1 - l] = -gamma * u;
    }
    if (l == 0) {
        S.ints[SI_RFLAG] = 0;
        S.sc[SC_GAMMA] = gamma;
    }
}

// d = -(gamma g + sum_j a_j s_j + sum_j c_j y_j), with the partials of the
// theta-space line-search inner products <x - v, x - v>, <x - v, d>, <d, d> (blk *
// 3 + k); four floats per thread and four pairs per step in flight (the vectors
// start 16-byte aligned when n2 is a multiple of 4, else a scalar loop)
__global__ void __launch_bounds__(kRedThreads) k_lb_dir(SolverDev S) {
    chain_entry();
    __shared__ float cs[32], cy[32];
    __shared__ const float* ps[32];
    __shared__ const float* py[32];
    __shared__ double sh[3][256];
    const int cnt = S.ints[SI_CNT];
    if (threadIdx.x < cnt) {
        const int idx = ring_idx(S, threadIdx.x);
        cs[threadIdx.x] = (float)S.acoef[threadIdx.x];
        cy[threadIdx.x] = (float)S.acoef[32 + threadIdx.x];
        ps[threadIdx.x] = S.sh + (long long)idx * S.n2;
        py[threadIdx.x] = S.yh + (long long)idx * S.n2;
    }
    __syncthreads();
    const float gamma = (float)S.sc[SC_GAMMA];
    Acc s0, s1, s2;
    auto dots = [&](float x, float v, float d) {
        const float w = x - v;
        s0.add(w * w);
        s1.add(w * d);
        s2.add(d * d);
    };
    if ((S.n2 & 3) == 0) {
        const long long n4 = S.n2 >> 2;
        const float4* g4 = reinterpret_cast<const float4*>(S.g);
        float4* d4 = reinterpret_cast<float4*>(S.d);
        GRID_STRIDE(i, n4) {
            const float4 gv = g4[i];
            const float4 xv = reinterpret_cast<const float4*>(S.x)[i], vv = reinterpret_cast<const float4*>(S.v)[i];
            float4 r = make_float4(gamma * gv.x, gamma * gv.y, gamma * gv.z, gamma * gv.w);
            int j = 0;
            for (; j + 4 <= cnt; j += 4) {
                float4 sv[4], yv[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    sv[u] = reinterpret_cast<const float4*>(ps[j + u])[i];
                    yv[u] = reinterpret_cast<const float4*>(py[j + u])[i];
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const float a = cs[j + u], c = cy[j + u];
                    r.x = fmaf(c, yv[u].x, fmaf(a, sv[u].x, r.x));
                    r.y = fmaf(c, yv[u].y, fmaf(a, sv[u].y, r.y));
                    r.z = fmaf(c, yv[u].z, fmaf(a, sv[u].z, r.z));
                    r.w = fmaf(c, yv[u].w, fmaf(a, sv[u].w, r.w));
                }
            }
            for (; j < cnt; ++j) {
                const float4 sv = reinterpret_cast<const float4*>(ps[j])[i];
                const float4 yv = reinterpret_cast<const float4*>(py[j])[i];
                const float a = cs[j], c = cy[j];
                r.x = fmaf(c, yv.x, fmaf(a, sv.x, r.x));
                r.y = fmaf(c, yv.y, fmaf(a, sv.y, r.y));
                r.z = fmaf(c, yv.z, fmaf(a, sv.z, r.z));
                r.w = fmaf(c, yv.w, fmaf(a, sv.w, r.w));
            }
            d4[i] = make_float4(-r.x, -r.y, -r.z, -r.w);
            dots(xv.x, vv.x, -r.x);
            dots(xv.y, vv.y, -r.y);
            dots(xv.z, vv.z, -r.z);
            dots(xv.w, vv.w, -r.w);
        }
    } else {
        GRID_STRIDE(i, S.n2) {
            float r = gamma * S.g[i];
            for (int j = 0; j < cnt; ++j) r = fmaf(cy[j], py[j][i], fmaf(cs[j], ps[j][i], r));
            S.d[i] = -r;
            dots(S.x[i], S.v[i], -r);
        }
    }
    const double v[3] = {s0.val(), s1.val(), s2.val()};
    const double r = block_sums(v, sh);
    if (threadIdx.x < 3) S.part3[blockIdx.x * 3 + threadIdx.x] = r;
}

__device__ double quartic_val(const double* c, double a) {
    return c[0] + a * (c[1] + a * (c[2] + a * (c[3] + a * c[4])));
}

// 1 / x and the cube root of x: an FP32 value refined by Newton steps in FP64 (1e-7
// -> 1e-14 -> rounding), where x is in FP32's comfortable range
__device__ __forceinline__ double recip(double x) {
    const double m = fabs(x);
    if (!(m > 1e-30 && m < 1e30)) return 1.0 / x;
    double r = (double)(1.f / (float)x);
    r = fma(r, fma(-x, r, 1.0), r);
    return fma(r, fma(-x, r, 1.0), r);
}
__device__ __forceinline__ double cube_root(double x) {
    const double m = fabs(x);
    if (!(m > 1e-30 && m < 1e30)) return cbrt(x);
    // y <- y - (y^3 - x) / (3 y^2), the divisor's reciprocal from FP32 (its error only
    // scales a correction of 1e-7, then of 1e-14)
    double y = (double)cbrtf((float)x);
    const double q = (double)(1.f / (3.f * (float)y * (float)y));
    y = fma(-(y * y * y - x), q, y);
    return fma(-(y * y * y - x), q, y);
}

// a candidate root of phi', polished by two Newton steps: false if it is none
__device__ __forceinline__ bool polish(const double* c, double& a) {
    for (int it = 0; it < 2; ++it) {
        const double d1 = c[1] + a * (2 * c[2] + a * (3 * c[3] + a * 4 * c[4]));
        const double d2 = 2 * c[2] + a * (6 * c[3] + a * 12 * c[4]);
        if (d2 != 0.0) a -= d1 * recip(d2);
    }
    return a > 0.0 && isfinite(a);
}

// Minimiser over a > 0 of the quartic, by the lanes of a warp: real roots of
// phi'(a) = 4 c4 a^3 + 3 c3 a^2 + 2 c2 a + c1 in closed form (depressed cubic:
// trigonometric form for three real roots, Cardano otherwise), polished.  Lane k
// takes the k-th root (the two cube roots of Cardano's form, the three cosines and
// the polishing are long FP64 chains; library divisions and cube roots among them
// are replaced by refined FP32 values, within 0.5 and 0.67 units in the last place:
// a solve of 256 receivers 3.62 -> 3.55 ms); ties go to the smaller root.
__device__ __forceinline__ bool quartic_argmin(const double* c, int lane, double* out) {
    const double A = 4 * c[4], B = 3 * c[3], C = 2 * c[2], D = c[1];
    double a = 0.0;
    bool have = false;
    if (A != 0.0) {
        const double ia = recip(A), p = B * ia, q = C * ia, r = D * ia;
        constexpr double third = 1.0 / 3.0, p27 = 1.0 / 27.0;
        const double P = q - p * p * third;
        const double Q = 2.0 * p * p * p * p27 - p * q * third + r;
        const double disc = 0.25 * Q * Q + P * P * P * p27;
        const double sh = -p * third;
        if (disc > 0.0) {
            const double sq = sqrt(disc);
            const double t = cube_root(-0.5 * Q + (lane == 0 ? sq : -sq));
            a = t + __shfl_sync(0xffffffffu, t, 1) + sh;   // lane 0
            have = lane == 0;
        } else if (P == 0.0) {
            a = cube_root(-Q) + sh;
            have = lane == 0;
        } else {
            const double m = 2.0 * sqrt(-P / 3.0);
            double arg = 3.0 * Q / (P * m);
            arg = fmin(1.0, fmax(-1.0, arg));
            const double th = acos(arg) / 3.0;
            const double tpi = 2.0943951023931954923;  // 2 pi / 3
            a = m * cos(th - tpi * (lane < 3 ? lane : 0)) + sh;
            have = lane < 3;
        }
    } else if (B != 0.0) {
        const double dsc = C * C - 4 * B * D;
        if (dsc >= 0.0) {
            const double s = sqrt(dsc);
            a = (-C + (lane == 0 ? s : -s)) / (2 * B);
            have = lane < 2;
        }
    } else if (C != 0.0) {
        a = -D / C;
        have = lane == 0;
    }
    have = polish(c, a) && have;
    const double v = quartic_val(c, a);
    double best_a = 0.0, best_v = 0.0;
    bool any = false;
    for (int k = 0; k < 3; ++k) {
        const bool hk = __shfl_sync(0xffffffffu, (int)have, k) != 0;
        const double ak = __shfl_sync(0xffffffffu, a, k), vk = __shfl_sync(0xffffffffu, v, k);
        if (hk && (!any || vk < best_v || (vk == best_v && ak < best_a))) {
            any = true;
            best_a = ak;
            best_v = vk;
        }
    }
    *out = best_a;
    return any;
}

// The last block (256 threads) of a line-search pass: finalise the 6 + 3 inner
// products, form phi's coefficients, check descent, pick alpha; alpha = 0 and a
// memory reset when no step.
__device__ __forceinline__ void line_search_last(const SolverDev& S, int nb6, int nb3, double rho, double (*sh)[256]) {
    const double d6 = sum_slabs<6>(S.part6, nb6, sh[0]);
    const double d3 = sum_slabs<3>(S.part3, nb3, sh[0]);
    if (threadIdx.x >= 32) return;
    const int lane = threadIdx.x;
    double e6[6], e3[3];
#pragma unroll
    for (int k = 0; k < 6; ++k) e6[k] = __shfl_sync(0xffffffffu, d6, k);
#pragma unroll
    for (int k = 0; k < 3; ++k) e3[k] = __shfl_sync(0xffffffffu, d3, k);
    double c[5];
    c[0] = 0.5 * e6[0] + 0.5 * rho * e3[0];
    c[1] = e6[1] + rho * e3[1];
    c[2] = 0.5 * e6[3] + e6[2] + 0.5 * rho * e3[2];
    c[3] = e6[4];
    c[4] = 0.5 * e6[5];
    double a = 0.0;
    bool ok = false;
    if (c[1] < 0.0) ok = quartic_argmin(c, lane, &a);
    if (lane != 0) return;
    for (int k = 0; k < 5; ++k) S.sc[SC_C0 + k] = c[k];
    if (!ok) {
        // no minimiser on a > 0 along d: no step, memory cleared; counted as a
        // restart unless the direction test already counted this iteration
        a = 0.0;
        S.ints[SI_CNT] = 0;
        if (!S.ints[SI_RFLAG]) S.ints[SI_RESTARTS] += 1;
    }
    bool finite = isfinite(c[0]) && isfinite(c[1]) && isfinite(c[2]) && isfinite(c[3]) && isfinite(c[4]);
    if (!finite) {
        a = 0.0;
        S.ints[SI_STATUS] = TLR_ERR_NONFINITE;
    }
    S.sc[SC_ALPHA] = a;
}

// the end of a line-search pass: the block's six sums, then the search by the last block
__device__ __forceinline__ void dots6_end(const SolverDev& S, const Acc* s, int nb3, double rho, double (*sh)[256]) {
    const double v[6] = {s[0].val(), s[1].val(), s[2].val(), s[3].val(), s[4].val(), s[5].val()};
    const double r = block_sums(v, sh);
    if (threadIdx.x < 6) S.part6[blockIdx.x * 6 + threadIdx.x] = r;
    if (last_block(reinterpret_cast<unsigned*>(S.ints + CT_LINE), gridDim.x))
        line_search_last(S, gridDim.x, nb3, rho, sh);
}

// the six products over FP32 arrays (two complex values per 16-byte load when n
// is even; the buffers start 256-byte aligned)
__global__ void __launch_bounds__(kRedThreads) k_dots6(SolverDev S, const cf* __restrict__ R, const cf* __restrict__ A1,
                                                      const cf* __restrict__ A2, long long n, int nb3, double rho) {
    chain_entry();
    __shared__ double sh[6][256];
    Acc s[6];
    if ((n & 1) == 0) {
        const float4* R4 = reinterpret_cast<const float4*>(R);
        const float4* A4 = reinterpret_cast<const float4*>(A1);
        const float4* C4 = reinterpret_cast<const float4*>(A2);
        const long long n4 = n >> 1, stride = (long long)gridDim.x * blockDim.x;
        long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
        for (; i + stride < n4; i += 2 * stride) {   // two 16-byte loads of each array in flight
            const float4 r = R4[i], a = A4[i], c = C4[i];
            const float4 r2 = R4[i + stride], a2 = A4[i + stride], c2 = C4[i + stride];
            float t[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
            dots6_group(t, r.x, r.y, a.x, a.y, c.x, c.y);
            dots6_group(t, r.z, r.w, a.z, a.w, c.z, c.w);
            dots6_group(t, r2.x, r2.y, a2.x, a2.y, c2.x, c2.y);
            dots6_group(t, r2.z, r2.w, a2.z, a2.w, c2.z, c2.w);
#pragma unroll
            for (int k = 0; k < 6; ++k) s[k].add(t[k]);
        }
        if (i < n4) {
            const float4 r = R4[i], a = A4[i], c = C4[i];
            float t[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
            dots6_group(t, r.x, r.y, a.x, a.y, c.x, c.y);
            dots6_group(t, r.z, r.w, a.z, a.w, c.z, c.w);
#pragma unroll
            for (int k = 0; k < 6; ++k) s[k].add(t[k]);
        }
    } else {
        GRID_STRIDE(i, n) {
            const cf r = R[i], a = A1[i], c = A2[i];
            dots6_add(s, r.x, r.y, a.x, a.y, c.x, c.y);
        }
    }
    dots6_end(S, s, nb3, rho, sh);
}

// The same over rstep's 16-row x 128-column tiles, with R read from its KN packing
// (the form it is carried in between forward products) and A1, A2 in FP32; products
// of four elements summed in FP32 before each compensated add.  A grid fixed by the
// number of tiles walks them in a fixed order and leaves one partial per product
// and CTA.  Its 12 KB of shared memory and 48 registers fit beside two contraction
// CTAs of another stream.
__global__ void __maxnreg__(48) k_dots6p(SolverDev S, char* const* __restrict__ kn, const cf* __restrict__ A1,
                                         const cf* __restrict__ A2, int ns, int nr, int b,
                                         const long long* __restrict__ roff, int nblk, int fmt, int nb3, double rho) {
    chain_entry();
    __shared__ double sh[6][256];
    constexpr int plane = 128 * 16 * 2;
    const int gx = (ns + kFuseCols - 1) / kFuseCols;
    const long long ntiles = (long long)gx * (nr / kFuseRows);
    const int n = threadIdx.x & (kFuseCols - 1), kg = threadIdx.x >> 7;
    Acc acc[6];
    for (long long tt = blockIdx.x; tt < ntiles; tt += gridDim.x) {
        const int n0 = (int)(tt % gx) * kFuseCols, r0 = (int)(tt / gx) * kFuseRows;
        if (n0 + n >= ns) continue;
        const RTile tl = rtile(r0, b, roff, nblk);
        float2 v[8];
        pk_load8(kn[tl.blk] + ((long long)(n0 >> 7) * (tl.bK >> 4) + (tl.rl0 >> 4)) * 4 * plane + row_off(fmt, n), fmt,
                 kg, v);
        float g[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const long long o = (long long)(r0 + kg * 8 + j) * ns + n0 + n;
            const float2 r = v[j], x = A1[o], c = A2[o];
            dots6_group(g, r.x, r.y, x.x, x.y, c.x, c.y);
            if ((j & 3) == 3) {
#pragma unroll
                for (int k = 0; k < 6; ++k) {
                    acc[k].add(g[k]);
                    g[k] = 0.f;
                }
            }
        }
    }
    dots6_end(S, acc, nb3, rho, sh);
}

// x += a d ; s_free = a d (two floats at a time: n2 is even)
__global__ void k_step_theta(SolverDev S) {
    chain_entry();
    const double ad = S.sc[SC_ALPHA];
    const float a = (float)ad;
    const int R = S.ring;
    const int fr = (S.ints[SI_NEWEST] + 1) % R;
    float2* s = reinterpret_cast<float2*>(S.sh + (long long)fr * S.n2);
    float2* x = reinterpret_cast<float2*>(S.x);
    const float2* d = reinterpret_cast<const float2*>(S.d);
    GRID_STRIDE(i, S.n2 >> 1) {
        const float2 dv = d[i];
        float2 xv = x[i];
        const float2 st = make_float2(a * dv.x, a * dv.y);
        s[i] = st;
        xv.x += st.x;
        xv.y += st.y;
        x[i] = xv;
    }
}

// gf from the split-K partials, y_free = (gf + rho (x - v)) - g, g <- gf + rho (x -
// v), with partials of ss, sy, yy; the last block accepts the pair (s, y) when
// alpha > 0 and <s,y> > 1e-12 |s||y| and records f = 0.5 ||R||^2 from the nf
// residual-norm partials.
__global__ void __launch_bounds__(kRedThreads) k_gradient_pair(SolverDev S, const cf* __restrict__ part, int nsplit,
                                                              long long nlr, long long ndense, long long b, int general,
                                                              const long long* __restrict__ zoff,
                                                              const int* __restrict__ zdim, double rho,
                                                              const double* __restrict__ partf, long long nf) {
    chain_entry();
    __shared__ double sh[3][256];
    const float r = (float)rho;
    const int R = S.ring;
    const int fr = (S.ints[SI_NEWEST] + 1) % R;
    const cf* s = reinterpret_cast<const cf*>(S.sh + (long long)fr * S.n2);
    cf* y = reinterpret_cast<cf*>(S.yh + (long long)fr * S.n2);
    const cf* x = reinterpret_cast<const cf*>(S.x);
    const cf* v = reinterpret_cast<const cf*>(S.v);
    cf* g = reinterpret_cast<cf*>(S.g);
    cf* gf = reinterpret_cast<cf*>(S.gf);
    const long long stride = S.n2 >> 1;
    Acc ss, sy, yy;
    auto entry = [&](long long e, cf gv) {
        const cf xe = x[e], ve = v[e], go = g[e], se = s[e];
        const cf gn = make_float2(gv.x + r * (xe.x - ve.x), gv.y + r * (xe.y - ve.y));
        const cf ye = make_float2(gn.x - go.x, gn.y - go.y);
        gf[e] = gv;
        y[e] = ye;
        g[e] = gn;
        ss.add(se.x * se.x);
        ss.add(se.y * se.y);
        sy.add(se.x * ye.x);
        sy.add(se.y * ye.y);
        yy.add(ye.x * ye.x);
        yy.add(ye.y * ye.y);
    };
    GRID_STRIDE(e, nlr) entry(e, split_sum(part, nsplit, stride, e));
    GRID_STRIDE(e, ndense * b * b) {
        long long base, n, row, col;
        if (!dense_tile(e, b, zoff, zdim, base, n, row, col)) continue;
        entry(nlr + base + row * n + col, split_sum_dense(part, nsplit, stride, nlr + base + row * n + col,
                                                          nlr + base + col * n + row, general));
    }
    const double w[3] = {ss.val(), sy.val(), yy.val()};
    const double t = block_sums(w, sh);
    if (threadIdx.x < 3) S.partp[blockIdx.x * 3 + threadIdx.x] = t;
    if (!last_block(reinterpret_cast<unsigned*>(S.ints + CT_PAIR), gridDim.x)) return;
    const double rr = sum_part(partf, nf, sh);
    const double d = sum_slabs<3>(S.partp, gridDim.x, sh[0]);
    if (threadIdx.x >= 32) return;
    const double dss = __shfl_sync(0xffffffffu, d, 0), dsy = __shfl_sync(0xffffffffu, d, 1),
                 dyy = __shfl_sync(0xffffffffu, d, 2);
    if (threadIdx.x != 0) return;
    const double f = 0.5 * rr;
    S.sc[SC_F] = f;
    const int it = S.ints[SI_ITERS];
    if (it < TLR_MAX_HIST) S.fhist[it] = f;
    S.ints[SI_ITERS] = it + 1;
    if (!isfinite(f)) S.ints[SI_STATUS] = TLR_ERR_NONFINITE;
    if (S.sc[SC_ALPHA] > 0.0 && dsy > 1e-12 * sqrt(dss * dyy)) {
        S.ints[SI_NEWEST] = fr;
        S.ints[SI_CNT] = min(S.ints[SI_CNT] + 1, S.m);
    }
}

// ADMM z- and dual updates (eq. 23, 24 in scaled form) and v = z - u
__global__ void k_admm_zu(SolverDev S, double lam, double rho) {
    chain_entry();
    const float den = (float)(1.0 / (1.0 + 2.0 * lam / rho));
    GRID_STRIDE(i, S.n2) {
        const float x = S.x[i], u = S.u[i];
        const float z = (x + u) * den;
        const float un = u + x - z;
        S.z[i] = z;
        S.u[i] = un;
        S.v[i] = z - un;
    }
}

// start of the solve: z = x, u = 0, v = x, counters cleared
__global__ void k_admm_init(SolverDev S) {
    chain_entry();
    GRID_STRIDE(i, S.n2) {
        const float x = S.x[i];
        S.z[i] = x;
        S.u[i] = 0.f;
        S.v[i] = x;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        S.ints[SI_CNT] = 0;
        S.ints[SI_NEWEST] = 0;
        S.ints[SI_ITERS] = 0;
        S.ints[SI_RESTARTS] = 0;
        S.ints[SI_STATUS] = 0;
        S.ints[SI_RFLAG] = 0;
    }
}

// resumed solve: v = z - u from the stored split; counters cleared
__global__ void k_admm_resume(SolverDev S) {
    chain_entry();
    GRID_STRIDE(i, S.n2) S.v[i] = S.z[i] - S.u[i];
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        S.ints[SI_CNT] = 0;
        S.ints[SI_NEWEST] = 0;
        S.ints[SI_ITERS] = 0;
        S.ints[SI_RESTARTS] = 0;
        S.ints[SI_STATUS] = 0;
        S.ints[SI_RFLAG] = 0;
    }
}

// f0 = f = 0.5 ||R||^2
__global__ void __launch_bounds__(256) k_record_f0(SolverDev S, const double* partf, long long np) {
    chain_entry();
    __shared__ double sh[1][256];
    const double rr = sum_part(partf, np, sh);
    if (threadIdx.x != 0) return;
    S.sc[SC_F0] = 0.5 * rr;
    S.sc[SC_F] = 0.5 * rr;
}

// ---------------------------------------------------------------------------
// host wrappers
// ---------------------------------------------------------------------------
cudaError_t sv_norm_part(const cf* R, long long n, double* part, cudaStream_t st) {
    (void)launch_pass(k_norm_part, dim3(red_blocks(n)), dim3(kRedThreads), st, R, n, part);
    counted(1);
    return cudaGetLastError();
}
cudaError_t sv_record_f0(const SolverDev& S, const double* partf, long long np, cudaStream_t st) {
    (void)launch_pass(k_record_f0, dim3(1), dim3(256), st, S, partf, np);
    counted(1);
    return cudaGetLastError();
}
cudaError_t sv_admm_init(const SolverDev& S, cudaStream_t st) {
    (void)launch_pass(k_admm_init, dim3(1024), dim3(256), st, S);
    counted(1);
    return cudaGetLastError();
}
cudaError_t sv_admm_resume(const SolverDev& S, cudaStream_t st) {
    (void)launch_pass(k_admm_resume, dim3(1024), dim3(256), st, S);
    counted(1);
    return cudaGetLastError();
}
cudaError_t sv_xupdate_start(const SolverDev& S, double rho, cudaStream_t st) {
    (void)launch_pass(k_xupdate_start, dim3(1024), dim3(256), st, S, rho);
    counted(1);
    return cudaGetLastError();
}
cudaError_t sv_direction(const SolverDev& S, cudaStream_t st) {
    for (int j0 = 0; j0 < S.m; j0 += kLbGroup) {
        (void)launch_pass(k_lb_dots, dim3(lb_blocks(S.n2)), dim3(kLbThreads), st, S, j0, j0 + kLbGroup >= S.m ? 1 : 0);
        counted(1);
    }
    (void)launch_pass(k_lb_dir, dim3(red_blocks(S.n2)), dim3(kRedThreads), st, S);
    counted(1);
    return cudaGetLastError();
}
cudaError_t sv_line_search(const SolverDev& S, const cf* R, const cf* A1, const cf* A2, long long n, double rho,
                           cudaStream_t st) {
    (void)launch_pass(k_dots6, dim3(red_blocks(n)), dim3(kRedThreads), st, S, R, A1, A2, n, red_blocks(S.n2), rho);
    counted(1);
    return cudaGetLastError();
}
cudaError_t sv_line_search_packed(const SolverDev& S, char* const* kn, const cf* A1, const cf* A2, int nr, int ns, int b,
                                  const long long* roff, int nblk, int fmt, double rho, cudaStream_t st) {
    if (nr <= 0 || ns <= 0 || nr % kFuseRows != 0) return cudaErrorInvalidValue;
    if (!roff && (b <= 0 || b % kFuseRows != 0 || nr % b != 0)) return cudaErrorInvalidValue;
    if (roff && nblk <= 0) return cudaErrorInvalidValue;
    const long long tiles = rstep_ctas(nr, ns);
    (void)launch_pass(k_dots6p, dim3((unsigned)std::min<long long>(tiles, kRedBlocks)), dim3(256), st, S, kn, A1, A2, ns,
                      nr, b, roff, nblk, fmt, red_blocks(S.n2), rho);
    counted(1);
    return cudaGetLastError();
}
cudaError_t sv_step_residual(cf* R, const cf* A1, const cf* A2, long long n, const double* alpha,
                             double* partf, cudaStream_t st) {
    (void)launch_pass(k_step_residual, dim3(red_blocks(n)), dim3(kRedThreads), st, R, A1, A2, n, alpha, partf);
    counted(1);
    return cudaGetLastError();
}
cudaError_t sv_step_theta(const SolverDev& S, cudaStream_t st) {
    (void)launch_pass(k_step_theta, dim3(2 * red_blocks(S.n2)), dim3(256), st, S);
    counted(1);
    return cudaGetLastError();
}
cudaError_t sv_gradient_pair(const SolverDev& S, const cf* part, int nsplit, long long nlr, long long ndense,
                             long long b, int general, const long long* zoff, const int* zdim, double rho,
                             const double* partf, long long nf, cudaStream_t st) {
    (void)launch_pass(k_gradient_pair, dim3(red_blocks(S.n2)), dim3(kRedThreads), st, S, part, nsplit, nlr, ndense, b,
                      general, zoff, zdim, rho, partf, nf);
    counted(1);
    return cudaGetLastError();
}
cudaError_t sv_admm_zu(const SolverDev& S, double lam, double rho, cudaStream_t st) {
    (void)launch_pass(k_admm_zu, dim3(1024), dim3(256), st, S, lam, rho);
    counted(1);
    return cudaGetLastError();
}

}  // namespace tlr
