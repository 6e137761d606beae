// Benchmark solver of eq. (4): conjugate gradients on the normal equations
//   P(G P(Z)) + 2 lambda Z = P(D-hat^H U-hat),  G = D-hat^H D-hat,
// P Z = (Z + Z^T)/2, with the real inner product Re tr(A^H B).  From Z = 0
// every iterate, residual and direction is exactly symmetric (the right-hand
// side is, and each update is elementwise symmetric), so P(p) = p and one
// iteration is y = G p (a dense GEMM, launched by the caller) plus the passes
// here: Ap = P(y) + 2 lambda p with <p, Ap>, the step, and the new direction.
// Scalars live on the device (FP64); reductions run on fixed grids and sum in
// a fixed order.
#include "internal.h"
#include "pack.h"
#include "reduce.h"

namespace tlr {

namespace {

constexpr int CG_T = 32;   // transpose tile
constexpr int kSymBlocks = 912;   // 6 per SM: fixed grid -> fixed summation order

enum CgSlot { CG_RR = 0, CG_PAP, CG_ALPHA, CG_BETA, CG_BN, CG_DONE, CG_ITERS, CG_CTR };   // CG_CTR: block counter

// the n partials summed by one block (256 threads), in every thread
__device__ __forceinline__ double sum_fixed(const double* part, int n, double (*sh)[256]) {
    double v[1] = {0.0};
    double a1 = 0.0, a2 = 0.0, a3 = 0.0;   // four sums keep the loads in flight
    int i = threadIdx.x;
    for (; i + 768 < n; i += 1024) {
        v[0] += part[i];
        a1 += part[i + 256];
        a2 += part[i + 512];
        a3 += part[i + 768];
    }
    for (; i < n; i += 256) v[0] += part[i];
    v[0] = (v[0] + a1) + (a2 + a3);
    (void)block_sums(v, sh);
    return sh[0][0];
}

// out = P(y) + s2 * p (s2 = 2 lambda), or out = P(y) if p == nullptr; with p,
// the last block forms alpha = rr / <p, out>, 0 once converged (or for a
// non-positive curvature).  32 x 32 tiles: the tile and its mirror are read
// through shared memory, both coalesced; a fixed grid walks the tiles.
__global__ void __launch_bounds__(256) k_cg_sym(const cf* __restrict__ y, const cf* __restrict__ p, float s2,
                                                cf* __restrict__ out, int n, double* __restrict__ part,
                                                double* __restrict__ sc) {
    chain_entry();
    __shared__ cf t[CG_T][CG_T + 1];
    __shared__ double sh[1][256];
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;     // 8 rows per pass
    const int nt = (n + CG_T - 1) / CG_T;
    Acc acc;
    for (int e = blockIdx.x; e < nt * nt; e += gridDim.x) {
        const int bx = e % nt * CG_T, by = e / nt * CG_T;       // out tile rows by.., cols bx..
        cf m[4], u[4], q[4];
        // mirror tile: y[bx + r][by + c] -> t[c][r]
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int r = ty + 8 * j;
            const bool mi = bx + r < n && by + tx < n, in = by + r < n && bx + tx < n;
            const long long o = (long long)(by + r) * n + bx + tx;
            m[j] = mi ? y[(long long)(bx + r) * n + by + tx] : make_float2(0.f, 0.f);
            u[j] = in ? y[o] : make_float2(0.f, 0.f);
            q[j] = in && p ? p[o] : make_float2(0.f, 0.f);
        }
        __syncthreads();   // the previous tile has been read
#pragma unroll
        for (int j = 0; j < 4; ++j) t[tx][ty + 8 * j] = m[j];
        __syncthreads();
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int r = ty + 8 * j;
            if (by + r < n && bx + tx < n) {
                const cf v = t[r][tx];
                cf w = make_float2(0.5f * (u[j].x + v.x), 0.5f * (u[j].y + v.y));
                if (p) {
                    w.x = fmaf(s2, q[j].x, w.x);
                    w.y = fmaf(s2, q[j].y, w.y);
                    acc.add(fmaf(q[j].x, w.x, q[j].y * w.y));
                }
                out[(long long)(by + r) * n + bx + tx] = w;
            }
        }
    }
    if (!p) return;
    const double v[1] = {acc.val()};
    const double s = block_sums(v, sh);
    if (threadIdx.x == 0) part[blockIdx.x] = s;
    if (!last_block(reinterpret_cast<unsigned*>(sc + CG_CTR), gridDim.x)) return;
    const double pap = sum_fixed(part, gridDim.x, sh);
    if (threadIdx.x == 0) {
        sc[CG_PAP] = pap;
        const bool go = sc[CG_DONE] == 0.0 && pap > 0.0 && isfinite(pap);
        sc[CG_ALPHA] = go ? sc[CG_RR] / pap : 0.0;
        if (!go) sc[CG_DONE] = 1.0;
    }
}

// r -= alpha Ap with ||r||^2; the last block forms beta = rr_new / rr and tests
// the convergence, or (init, Ap == nullptr) sets rr = ||b||^2 = ||r||^2
__global__ void __launch_bounds__(kRedThreads) k_cg_step(cf* __restrict__ r, const cf* __restrict__ Ap, long long n2,
                                                         double tol, double* __restrict__ sc,
                                                         double* __restrict__ part) {
    chain_entry();
    __shared__ double sh[1][256];
    const float a = Ap ? (float)sc[CG_ALPHA] : 0.f;
    Acc acc;
    const long long stride = (long long)gridDim.x * blockDim.x;
    const long long n4 = n2 >> 1;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n4; i += stride) {
        float4 ri = reinterpret_cast<const float4*>(r)[i];
        if (a != 0.f) {
            const float4 q = reinterpret_cast<const float4*>(Ap)[i];
            ri.x = fmaf(-a, q.x, ri.x);
            ri.y = fmaf(-a, q.y, ri.y);
            ri.z = fmaf(-a, q.z, ri.z);
            ri.w = fmaf(-a, q.w, ri.w);
            reinterpret_cast<float4*>(r)[i] = ri;
        }
        acc.add(fmaf(ri.x, ri.x, ri.y * ri.y));
        acc.add(fmaf(ri.z, ri.z, ri.w * ri.w));
    }
    if ((n2 & 1) && blockIdx.x == 0 && threadIdx.x == 0) {   // an odd number of values: the last one
        cf ri = r[n2 - 1];
        if (a != 0.f) {
            ri.x = fmaf(-a, Ap[n2 - 1].x, ri.x);
            ri.y = fmaf(-a, Ap[n2 - 1].y, ri.y);
            r[n2 - 1] = ri;
        }
        acc.add(fmaf(ri.x, ri.x, ri.y * ri.y));
    }
    const double v[1] = {acc.val()};
    const double s = block_sums(v, sh);
    if (threadIdx.x == 0) part[blockIdx.x] = s;
    if (!last_block(reinterpret_cast<unsigned*>(sc + CG_CTR), gridDim.x)) return;
    const double rn = sum_fixed(part, gridDim.x, sh);
    if (threadIdx.x != 0) return;
    if (!Ap) {
        sc[CG_RR] = rn;
        sc[CG_BN] = rn;
        sc[CG_DONE] = rn > 0.0 ? 0.0 : 1.0;
        sc[CG_ITERS] = 0.0;
    } else if (sc[CG_ALPHA] != 0.0) {
        sc[CG_BETA] = rn / sc[CG_RR];
        sc[CG_RR] = rn;
        sc[CG_ITERS] += 1.0;
        if (!(rn > tol * tol * sc[CG_BN])) sc[CG_DONE] = 1.0;
    } else {
        sc[CG_BETA] = 0.0;
    }
}

// x += alpha p, p = r + beta p (skipped once converged), and p as the next
// product's packed B operand (pk != nullptr; p is symmetric, its rows serve).
// A warp takes 16 rows x 16 columns, one packed 16-row group: 8 lanes read a
// row's 128 bytes, two values each, and their BF16 pairs fill 64 contiguous
// bytes of each plane (thread = 8 columns of a row, 16-byte stores: 55 us
// at n = 2048, the reads touching 16 lines per instruction).
__global__ void __launch_bounds__(256) k_cg_dir(cf* __restrict__ x, cf* __restrict__ p, const cf* __restrict__ r,
                                                int n, const double* __restrict__ sc, char* __restrict__ pk) {
    chain_entry();
    if (sc[CG_ALPHA] == 0.0) return;   // converged earlier: p and its packing stand
    const float al = (float)sc[CG_ALPHA], be = (float)sc[CG_BETA];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int c = blockIdx.x * 16 + (lane & 7) * 2;
    if (c >= n) return;   // the packing's padding stays zero
    const bool vec = (n & 1) == 0 && (reinterpret_cast<uintptr_t>(x) & 15) == 0;   // x is the caller's buffer
    const int nkc = (n + 15) >> 4;
    char* const tile = pk + ((long long)blockIdx.y * nkc + blockIdx.x) * kPackTile;
    float4 rv[4], pv[4], xv[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int row = blockIdx.y * 128 + warp * 16 + i * 4 + (lane >> 3);
        const long long o = (long long)row * n + c;
        rv[i] = pv[i] = xv[i] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (row < n) {
            if (vec) {
                rv[i] = *reinterpret_cast<const float4*>(r + o);
                pv[i] = *reinterpret_cast<const float4*>(p + o);
                xv[i] = *reinterpret_cast<const float4*>(x + o);
            } else {
                const cf a = r[o], b = p[o], d = x[o];
                rv[i].x = a.x, rv[i].y = a.y, pv[i].x = b.x, pv[i].y = b.y, xv[i].x = d.x, xv[i].y = d.y;
                if (c + 1 < n) {
                    const cf a1 = r[o + 1], b1 = p[o + 1], d1 = x[o + 1];
                    rv[i].z = a1.x, rv[i].w = a1.y, pv[i].z = b1.x, pv[i].w = b1.y, xv[i].z = d1.x, xv[i].w = d1.y;
                }
            }
        }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int rl = warp * 16 + i * 4 + (lane >> 3), row = blockIdx.y * 128 + rl;
        if (row >= n) continue;
        const long long o = (long long)row * n + c;
        float4 q = pv[i], t = xv[i];
        t.x = fmaf(al, q.x, t.x);
        t.y = fmaf(al, q.y, t.y);
        t.z = fmaf(al, q.z, t.z);
        t.w = fmaf(al, q.w, t.w);
        q.x = fmaf(be, q.x, rv[i].x);
        q.y = fmaf(be, q.y, rv[i].y);
        q.z = fmaf(be, q.z, rv[i].z);
        q.w = fmaf(be, q.w, rv[i].w);
        if (vec) {
            *reinterpret_cast<float4*>(x + o) = t;
            *reinterpret_cast<float4*>(p + o) = q;
        } else {
            x[o] = make_float2(t.x, t.y);
            p[o] = make_float2(q.x, q.y);
            if (c + 1 < n) {
                x[o + 1] = make_float2(t.z, t.w);
                p[o + 1] = make_float2(q.z, q.w);
            }
        }
        if (pk)
            pk_store2(tile + row_off(kFmtBF16X3, rl), kFmtBF16X3, lane & 7, make_float2(q.x, q.y), make_float2(q.z, q.w));
    }
}

}  // namespace

int cg_partials() { return std::max(kSymBlocks, kRedBlocks); }

cudaError_t cg_sym(const cf* y, const cf* p, float s2, cf* out, int n, double* part, double* sc, cudaStream_t st) {
    const int t = (n + CG_T - 1) / CG_T;
    counted(1);
    return launch_chain(k_cg_sym, dim3(std::min(t * t, kSymBlocks)), dim3(256), 0, st, y, p, s2, out, n, part, sc);
}

// start: x = 0, r = p = b (r holds b on entry), sc cleared, rr = ||b||^2
cudaError_t cg_start(cf* x, cf* r, cf* p, int n, double* part, double* sc, cudaStream_t st) {
    const long long n2 = (long long)n * n;
    cudaError_t e = cudaMemsetAsync(x, 0, n2 * sizeof(cf), st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(p, r, n2 * sizeof(cf), cudaMemcpyDeviceToDevice, st);
    if (e == cudaSuccess) e = cudaMemsetAsync(sc, 0, 8 * sizeof(double), st);
    if (e != cudaSuccess) return e;
    counted(1);
    return launch_chain(k_cg_step, dim3(kRedBlocks), dim3(kRedThreads), 0, st, r, (const cf*)nullptr, n2, 0.0, sc, part);
}

cudaError_t cg_iteration_tail(cf* x, cf* r, cf* p, const cf* Ap, int n, double tol, double* part, double* sc, char* pk,
                              cudaStream_t st) {
    const long long n2 = (long long)n * n;
    counted(2);
    const cudaError_t e = launch_chain(k_cg_step, dim3(kRedBlocks), dim3(kRedThreads), 0, st, r, Ap, n2, tol, sc, part);
    if (e != cudaSuccess) return e;
    return launch_chain(k_cg_dir, dim3((n + 15) / 16, (n + 127) / 128), dim3(256), 0, st, x, p, (const cf*)r, n,
                        (const double*)sc, pk);
}

}  // namespace tlr
