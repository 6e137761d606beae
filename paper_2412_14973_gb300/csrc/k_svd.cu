// Tile singular value decompositions for the hyper-parameter selection and
// warm start (the tile rank rule and the SVD / Takagi initialisation).
//
// One CTA per m x n tile of a dense nr x nr matrix (row-major): one-sided
// (Hestenes) Jacobi on the tile's n columns, complex FP32.  A sweep visits
// every column pair once in round-robin order (n - 1 rounds of n/2 disjoint
// pairs, one warp per pair); a pair (p, q) with Gram entries alpha = |a_p|^2,
// beta = |a_q|^2, gamma = a_p^H a_q is made orthogonal by the unitary
// [a_p, a_q e^{-i phi}] [[c, s], [-s, c]], phi = arg gamma, t = s / c the
// smaller root of t^2 + 2 zeta t - 1 = 0, zeta = (beta - alpha) / (2 |gamma|);
// V accumulates the same column operations.  Sweeps stop once every pair has
// |gamma| <= tol sqrt(alpha beta) (or after max_sweeps): then
// A_0 = U Sigma V^H with sigma_c = |a_c| and u_c = a_c / sigma_c (columns that
// end at zero, n - m of them at least when n > m, have sigma_c = 0).
//
// What bounds it: instruction issue -- per pair the sums and rotation of 2 m
// values, and a scalar part (five square roots, four divisions) that a warp per
// pair spends on 32 lanes.  So a warp takes P pairs at a time: their 4 P sums go
// down one butterfly that halves the values per lane at each step (16 shuffles
// for 4 pairs instead of 80; the same tree of additions), the scalar parts run
// side by side in groups of lanes, and each pair's two columns stay in registers
// from the sums to the rotation.  As many columns of A, then of V, as fit live in
// shared memory (all of A and 94 of V's 128 columns for a 128 x 128 tile; 111 of
// A's for 256 x 256), the rest in global memory (L2).  With a warp per pair,
// every column in L2 and read twice, 78 tiles of 128 x 128 took 8.2 ms (singular
// values) and 9.5 ms (with V); now 5.3 and 7.1 (256 x 256, 136 tiles, values only:
// 52.6 and 37.1).  The order of pairs, sums and
// operations does not depend on P or on where a column lives, and the products
// that are fused are written out, so the results are the same bits.
#include <algorithm>

#include "internal.h"

namespace tlr {

namespace {

constexpr int SVD_SMEM = 222 * 1024;   // columns of A and V in shared memory, at most

constexpr int SVD_THREADS = 512;       // at most; 128 registers

__device__ __forceinline__ float warp_sumf(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// player at position m of round r (circle method; position 0 is fixed):
// ((m - 1 + r) mod (nb - 1)) + 1 with m, r < nb
__device__ __forceinline__ int player(int m, int r, int nb) {
    const int i = m + r;
    return m == 0 ? 0 : (i > nb - 1 ? i - (nb - 1) : i);
}

// two FP32 operations per instruction, on (re, im) pairs
typedef unsigned long long f2;
__device__ __forceinline__ f2 pack2(float x, float y) {
    f2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(x), "f"(y));
    return r;
}
__device__ __forceinline__ float2 unpack2(f2 a) {
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(a));
    return r;
}
__device__ __forceinline__ f2 mul2(f2 a, f2 b) {
    f2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c) {
    f2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}

// The rotation of one pair of values by (c, s) and the phase (er, ei); the first
// product of each sum is the fused one:
//   b = y (er + i ei),  x <- c x - s b,  y <- s x + c b
__device__ __forceinline__ void rotate(f2& x, f2& y, f2 cc, f2 ss, f2 ns, f2 e, f2 ie) {
    const float2 v = unpack2(y);
    const f2 b = fma2(pack2(v.x, v.x), e, mul2(pack2(v.y, v.y), ie));   // e = (er, ei), ie = (-ei, er)
    y = fma2(ss, x, mul2(cc, b));
    x = fma2(cc, x, mul2(ns, b));
}

// R = ceil(max rows / 32): values of a column per lane; P pairs per warp (1, 2
// or 4)
template <int R, int P>
__global__ void __launch_bounds__(SVD_THREADS) k_tile_svd(const cf* __restrict__ X, long long ldx,
                                                          const SvdTile* __restrict__ tiles, int bmax,
                                                          cf* __restrict__ work, int want_vec, int max_sweeps,
                                                          float tol, float* __restrict__ sig,
                                                          int* __restrict__ order, int* __restrict__ sweeps_out,
                                                          int smem_bytes) {
    extern __shared__ __align__(16) cf cols[];
    const int t = blockIdx.x;
    const SvdTile tg = tiles[t];
    // the matrix the sweeps work on: the tile (m x n) or its transpose
    const int m = tg.trans ? tg.n : tg.m, n = tg.trans ? tg.m : tg.n, nb = n + (n & 1);
    const long long slot = (long long)bmax * bmax;
    cf* const Ag = work + (long long)t * (want_vec ? 2 : 1) * slot;   // column-major m x n
    cf* const Vg = Ag + slot;                                         // column-major n x n
    // columns in shared memory: the first sa of A, then the first sv of V
    const int room = smem_bytes / (int)sizeof(cf);
    const int sa = min(n, room / m), sv = want_vec ? min(n, (room - sa * m) / n) : 0;
    cf* const Vs = cols + sa * m;
    auto colA = [&](int c) { return c < sa ? cols + c * m : Ag + (long long)c * m; };
    auto colV = [&](int c) { return c < sv ? Vs + c * n : Vg + (long long)c * n; };
    __shared__ unsigned int smax;
    __shared__ float snorm[512];
    // load the tile (reads coalesced along the rows of X), V = I
    for (int e = threadIdx.x; e < m * n; e += blockDim.x) {
        if (tg.trans) {
            const int r = e % m, c = e / m;   // A[r][c] = X tile[c][r]
            colA(c)[r] = X[((long long)tg.r0 + c) * ldx + (long long)tg.c0 + r];
        } else {
            const int r = e / n, c = e % n;
            colA(c)[r] = X[((long long)tg.r0 + r) * ldx + (long long)tg.c0 + c];
        }
    }
    if (want_vec)
        for (int e = threadIdx.x; e < n * n; e += blockDim.x)
            colV(e / n)[e % n] = make_float2((e / n) == (e % n) ? 1.f : 0.f, 0.f);
    __syncthreads();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nwarp = blockDim.x >> 5;
    constexpr int NV = 4 * P, GRP = 32 / P;   // sums of a batch; lanes per pair in the scalar part
    int sw = 0;
    for (; sw < max_sweeps; ++sw) {
        if (threadIdx.x == 0) smax = 0u;
        __syncthreads();
        float mx = 0.f;
        for (int r = 0; r < nb - 1; ++r) {
            for (int k0 = warp * P; k0 < nb / 2; k0 += nwarp * P) {
                f2 x[P][R], y[P][R];
                f2 *ap[P], *aq[P];
                int pp[P], qq[P];
                float sum[NV];   // |a_p|^2, |a_q|^2, Re and Im of a_p^H a_q of each pair
#pragma unroll
                for (int u = 0; u < P; ++u) {
                    const int k = k0 + u;
                    const int p = player(k, r, nb), q = player(nb - 1 - k, r, nb);
                    const bool on = k < nb / 2 && p < n && q < n;   // not the dummy player of an odd n
                    pp[u] = on ? p : 0;
                    qq[u] = on ? q : 0;
                    ap[u] = reinterpret_cast<f2*>(colA(pp[u]));
                    aq[u] = reinterpret_cast<f2*>(colA(qq[u]));
#pragma unroll
                    for (int j = 0; j < R; ++j) {
                        const int i = lane + 32 * j;
                        x[u][j] = on && i < m ? ap[u][i] : 0;
                        y[u][j] = on && i < m ? aq[u][i] : 0;
                    }
                }
#pragma unroll
                for (int u = 0; u < P; ++u) {
                    float al = 0.f, be = 0.f;
                    f2 gg = 0;   // Re and Im of conj(x) y
#pragma unroll
                    for (int j = 0; j < R; ++j) {
                        const float2 v = unpack2(x[u][j]), w = unpack2(y[u][j]);
                        al = fmaf(v.x, v.x, fmaf(v.y, v.y, al));
                        be = fmaf(w.x, w.x, fmaf(w.y, w.y, be));
                        gg = fma2(pack2(v.x, v.x), y[u][j], fma2(pack2(v.y, -v.y), pack2(w.y, w.x), gg));
                    }
                    sum[4 * u] = al;
                    sum[4 * u + 1] = be;
                    sum[4 * u + 2] = unpack2(gg).x;
                    sum[4 * u + 3] = unpack2(gg).y;
                }
                // butterfly over the lanes; while more than one value is left, a
                // lane keeps the half that its bit says and sends the other
                int left = NV;
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) {
                    if (left > 1) {
                        left >>= 1;
                        const bool hi = (lane & o) != 0;
#pragma unroll
                        for (int v = 0; v < NV / 2; ++v)
                            if (v < left) {
                                const float keep = hi ? sum[v + left] : sum[v], send = hi ? sum[v] : sum[v + left];
                                sum[v] = keep + __shfl_xor_sync(0xffffffffu, send, o);
                            }
                    } else {
                        sum[0] += __shfl_xor_sync(0xffffffffu, sum[0], o);
                    }
                }
                // the lane group of pair u: lanes u GRP ..; kind t in its quarter t
                const int g0 = lane & ~(GRP - 1);
                const float al = __shfl_sync(0xffffffffu, sum[0], g0);
                const float be = __shfl_sync(0xffffffffu, sum[0], g0 + GRP / 4);
                const float gr = __shfl_sync(0xffffffffu, sum[0], g0 + GRP / 2);
                const float gi = __shfl_sync(0xffffffffu, sum[0], g0 + 3 * GRP / 4);
                const float g = sqrtf(fmaf(gr, gr, __fmul_rn(gi, gi)));
                const bool turn = al > 0.f && be > 0.f && g > tol * sqrtf(al) * sqrtf(be);
                const unsigned turns = __ballot_sync(0xffffffffu, turn);
                if (turns == 0) continue;
                float c = 1.f, s = 0.f, er = 1.f, ei = 0.f;
                if (turn) {
                    mx = fmaxf(mx, g / (sqrtf(al) * sqrtf(be)));
                    const float zeta = (be - al) / (2.f * g);
                    const float tt = (zeta >= 0.f ? 1.f : -1.f) / (fabsf(zeta) + sqrtf(fmaf(zeta, zeta, 1.f)));
                    c = rsqrtf(fmaf(tt, tt, 1.f));
                    s = c * tt;
                    er = gr / g;
                    ei = -gi / g;   // e^{-i phi}
                }
                // the pairs' rotations, from their lane groups to the warp
                f2 cc[P], ss[P], e[P];
#pragma unroll
                for (int u = 0; u < P; ++u) {
                    const float cu = __shfl_sync(0xffffffffu, c, u * GRP), su = __shfl_sync(0xffffffffu, s, u * GRP);
                    cc[u] = pack2(cu, cu);
                    ss[u] = pack2(su, su);
                    e[u] = pack2(__shfl_sync(0xffffffffu, er, u * GRP), __shfl_sync(0xffffffffu, ei, u * GRP));
                }
                auto turned = [&](int u) { return ((turns >> (u * GRP)) & 1) != 0; };
                auto turn_rows = [&](int u, f2* p, f2* q, int rows) {
                    const float2 ev = unpack2(e[u]);
                    const f2 ie = pack2(-ev.y, ev.x), ns = pack2(-unpack2(ss[u]).x, -unpack2(ss[u]).x);
#pragma unroll
                    for (int j = 0; j < R; ++j) {
                        const int i = lane + 32 * j;
                        rotate(x[u][j], y[u][j], cc[u], ss[u], ns, e[u], ie);
                        if (i < rows) {
                            p[i] = x[u][j];
                            q[i] = y[u][j];
                        }
                    }
                };
#pragma unroll
                for (int u = 0; u < P; ++u)
                    if (turned(u)) turn_rows(u, ap[u], aq[u], m);
                if (want_vec) {
#pragma unroll
                    for (int u = 0; u < P; ++u) {
                        if (!turned(u)) continue;
                        const f2* vp = reinterpret_cast<const f2*>(colV(pp[u]));
                        const f2* vq = reinterpret_cast<const f2*>(colV(qq[u]));
#pragma unroll
                        for (int j = 0; j < R; ++j) {
                            const int i = lane + 32 * j;
                            x[u][j] = i < n ? vp[i] : 0;
                            y[u][j] = i < n ? vq[i] : 0;
                        }
                    }
#pragma unroll
                    for (int u = 0; u < P; ++u)
                        if (turned(u))
                            turn_rows(u, reinterpret_cast<f2*>(colV(pp[u])), reinterpret_cast<f2*>(colV(qq[u])), n);
                }
            }
            __syncthreads();
        }
        if (mx > 0.f) atomicMax(&smax, __float_as_uint(mx));
        __syncthreads();
        if (__uint_as_float(smax) <= tol) {
            ++sw;
            break;
        }
        __syncthreads();
    }
    // sigma_c = |a_c|, then the order of decreasing sigma (ties by column);
    // slots n .. bmax-1 get sigma = -1 (below every threshold)
    for (int c = warp; c < n; c += nwarp) {
        const cf* ac = colA(c);
        float s2 = 0.f;
        for (int i = lane; i < m; i += 32) s2 = fmaf(ac[i].x, ac[i].x, fmaf(ac[i].y, ac[i].y, s2));
        s2 = warp_sumf(s2);
        if (lane == 0) snorm[c] = sqrtf(s2);
    }
    __syncthreads();
    for (int c = threadIdx.x; c < n; c += blockDim.x) {
        const float v = snorm[c];
        int rk = 0;
        for (int c2 = 0; c2 < n; ++c2) {
            const float w = snorm[c2];
            rk += (w > v) || (w == v && c2 < c);
        }
        sig[(long long)t * bmax + rk] = v;
        if (order) order[(long long)t * bmax + rk] = c;
    }
    for (int c = n + threadIdx.x; c < bmax; c += blockDim.x) {
        sig[(long long)t * bmax + c] = -1.f;
        if (order) order[(long long)t * bmax + c] = 0;
    }
    if (want_vec) {   // the columns kept in shared memory go where the warm start reads them
        for (int e = threadIdx.x; e < sa * m; e += blockDim.x) Ag[e] = cols[e];
        for (int e = threadIdx.x; e < sv * n; e += blockDim.x) Vg[e] = Vs[e];
    }
    if (threadIdx.x == 0 && sweeps_out) sweeps_out[t] = sw;
}

// one block: v0 = max sigma over all tiles; rank of tile t = #{sigma >= eps v0}
__global__ void k_rank_rule(const float* __restrict__ sig, int ntiles, int b, double eps, int* __restrict__ ranks,
                            double* __restrict__ v0_out) {
    __shared__ float smx[32];
    float m = 0.f;
    for (int t = threadIdx.x; t < ntiles; t += blockDim.x) m = fmaxf(m, sig[(long long)t * b]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0) smx[threadIdx.x >> 5] = m;
    __syncthreads();
    if (threadIdx.x < 32) {
        m = threadIdx.x < (blockDim.x >> 5) ? smx[threadIdx.x] : 0.f;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
        if (threadIdx.x == 0) smx[0] = m;
    }
    __syncthreads();
    const double v0 = smx[0];
    const float thr = (float)(eps * v0);
    for (int t = threadIdx.x; t < ntiles; t += blockDim.x) {
        int k = 0;
        while (k < b && sig[(long long)t * b + k] >= thr) ++k;
        ranks[t] = k;
    }
    if (threadIdx.x == 0) *v0_out = v0;
}

// Warm-start factors from tile SVDs (one CTA per tile, one thread per column
// q < k of the factor, rows in a loop):
//   low-rank tile (kind 0, m x n): L = U_k Sigma_k^1/2 (m x k), R = conj(V_k)
//     Sigma_k^1/2 (n x k), so L R^T = U_k Sigma_k V_k^H;
//   low-rank diagonal of the reciprocal form (kind 1, square): Q = conj(V_k)
//     E_k Sigma_k^1/2 with E = diag(V^T U)^1/2 (Takagi form of the symmetric
//     tile), Q Q^T = U_k Sigma_k V_k^H;
//   dense diagonal (kind 2): Z = the m x m tile itself (no SVD).
//   A tile whose SVD ran on its transpose (trans: T^T = U' Sigma V'^H) has
//   U = conj(V'), V = conj(U'): L = conj(V'_k) Sigma^1/2, R = U'_k Sigma^1/2.
__global__ void k_warm_fill(const cf* __restrict__ X, long long ldx, const WarmTile* __restrict__ wt, int bmax,
                            const cf* __restrict__ work, const float* __restrict__ sig,
                            const int* __restrict__ order, cf* __restrict__ theta) {
    const WarmTile w = wt[blockIdx.x];
    const int m = w.m, n = w.n;
    const int jm = w.trans ? n : m, jn = w.trans ? m : n;   // the SVD's rows and columns
    if (w.kind == 2) {
        for (long long e = threadIdx.x; e < (long long)m * m; e += blockDim.x) {
            const int r = (int)(e / m), c = (int)(e % m);
            theta[w.offL + e] = X[((long long)w.r0 + r) * ldx + (long long)w.c0 + c];
        }
        return;
    }
    const long long slot = (long long)bmax * bmax;
    const cf* A = work + (long long)w.svd * 2 * slot;   // column-major jm x jn
    const cf* V = A + slot;                             // column-major jn x jn
    for (int q = threadIdx.x; q < w.k; q += blockDim.x) {
        const int c = order[(long long)w.svd * bmax + q];
        const float s = sig[(long long)w.svd * bmax + q];
        const float rs = sqrtf(s), inv = s > 0.f ? 1.f / s : 0.f;
        const cf* ac = A + (long long)c * jm;
        const cf* vc = V + (long long)c * jn;
        if (w.kind == 0) {
            // u_c = a_c / s (jm rows), v_c (jn rows)
            cf* Lq = theta + w.offL + q;
            cf* Rq = theta + w.offR + q;
            if (!w.trans) {
                for (int r = 0; r < m; ++r) Lq[(long long)r * w.k] = make_float2(ac[r].x * inv * rs, ac[r].y * inv * rs);
                for (int r = 0; r < n; ++r) Rq[(long long)r * w.k] = make_float2(vc[r].x * rs, -vc[r].y * rs);
            } else {
                for (int r = 0; r < m; ++r) Lq[(long long)r * w.k] = make_float2(vc[r].x * rs, -vc[r].y * rs);
                for (int r = 0; r < n; ++r) Rq[(long long)r * w.k] = make_float2(ac[r].x * inv * rs, ac[r].y * inv * rs);
            }
        } else {
            // d = sum_r V[r] U[r] (U = a_c / s): the phase pair of the Takagi form
            float dr = 0.f, di = 0.f;
            for (int r = 0; r < m; ++r) {
                const cf u = ac[r], v = vc[r];
                dr = fmaf(v.x, u.x, fmaf(-v.y, u.y, dr));
                di = fmaf(v.x, u.y, fmaf(v.y, u.x, di));
            }
            const float ph = 0.5f * atan2f(di, dr);
            const float er = cosf(ph), ei = sinf(ph);
            for (int r = 0; r < m; ++r) {
                const cf v = vc[r];
                // conj(v) e^{i ph} sqrt(s)
                const float xr = v.x * er + v.y * ei, xi = v.x * ei - v.y * er;
                theta[w.offL + (long long)r * w.k + q] = make_float2(xr * rs, xi * rs);
            }
        }
    }
}

}  // namespace

size_t tile_svd_work_bytes(int ntiles, int b, bool vec) { return (size_t)ntiles * (vec ? 2 : 1) * b * b * sizeof(cf); }

cudaError_t tile_svd(const cf* X, long long ldx, const SvdTile* tiles, int ntiles, int bmax, cf* work, bool vec,
                     int max_sweeps, float tol, float* sig, int* order, int* sweeps, cudaStream_t st) {
    if (ntiles == 0) return cudaSuccess;
    if (bmax < 1 || bmax > 512) return cudaErrorInvalidValue;
    // shared memory for the columns of the largest tile (or what there is of it);
    // a warp per pair of a round
    const long long want = (long long)bmax * bmax * (vec ? 2 : 1) * (long long)sizeof(cf);
    const int smem = (int)std::min<long long>(want, SVD_SMEM);
    const int R = (bmax + 31) / 32, pairs = (bmax + 1) / 2;
#define TLR_SVD(Rv, Pv)                                                                                         \
    do {                                                                                                        \
        cudaError_t e =                                                                                         \
            cudaFuncSetAttribute(k_tile_svd<Rv, Pv>, cudaFuncAttributeMaxDynamicSharedMemorySize, SVD_SMEM);    \
        if (e != cudaSuccess) return e;                                                                         \
        k_tile_svd<Rv, Pv><<<ntiles, std::min(SVD_THREADS, 32 * ((pairs + Pv - 1) / Pv)), smem, st>>>(          \
            X, ldx, tiles, bmax, work, vec ? 1 : 0, max_sweeps, tol, sig, order, sweeps, smem);                 \
    } while (0)
    // P pairs of 2 R values per warp: 64 registers
    if (R <= 1)
        TLR_SVD(1, 4);
    else if (R <= 2)
        TLR_SVD(2, 4);
    else if (R <= 4)
        TLR_SVD(4, 4);
    else if (R <= 8)
        TLR_SVD(8, 2);
    else
        TLR_SVD(16, 1);
#undef TLR_SVD
    counted(1);
    return cudaGetLastError();
}

cudaError_t rank_rule(const float* sig, int ntiles, int b, double eps, int* ranks, double* v0, cudaStream_t st) {
    k_rank_rule<<<1, 256, 0, st>>>(sig, ntiles, b, eps, ranks, v0);
    counted(1);
    return cudaGetLastError();
}

cudaError_t warm_fill(const cf* X, long long ldx, const WarmTile* wt, int nt, int bmax, const cf* work,
                      const float* sig, const int* order, cf* theta, cudaStream_t st) {
    if (nt == 0) return cudaSuccess;
    k_warm_fill<<<nt, 128, 0, st>>>(X, ldx, wt, bmax, work, sig, order, theta);
    counted(1);
    return cudaGetLastError();
}

}  // namespace tlr
