// Data-preparation kernels: Hilbert receiver order (eq. 10), normalisation
// alpha (Hyper-parameter selection section), receiver-major reordered panels
// (eq. 14) and the natural-order back-mapping X = S X_h S^T (eq. 11).
#include <algorithm>

#include "internal.h"

namespace tlr {

// Distance of cell (x, y) along the Hilbert curve on an n x n square (n a
// power of two): quadrant (rx, ry) at level s contributes s*s*((3 rx) ^ ry)
// cells visited before it; the coordinates are then reflected / swapped so the
// sub-square is walked in the base orientation (0,0),(0,1),(1,1),(1,0).
__device__ __forceinline__ long long hilbert_d(long long n, long long x, long long y) {
    long long d = 0;
    for (long long s = n >> 1; s > 0; s >>= 1) {
        const int rx = (x & s) ? 1 : 0;
        const int ry = (y & s) ? 1 : 0;
        d += s * s * (long long)((3 * rx) ^ ry);
        if (ry == 0) {
            if (rx == 1) {
                x = n - 1 - x;
                y = n - 1 - y;
            }
            const long long t = x;
            x = y;
            y = t;
        }
    }
    return d;
}

// slot[key(r)] = r for every receiver; slot is n*n, pre-filled with -1.
__global__ void k_hilbert_scatter(int nx, int ny, long long n, int32_t* slot) {
    const long long nr = (long long)nx * ny;
    for (long long r = blockIdx.x * (long long)blockDim.x + threadIdx.x; r < nr;
         r += (long long)gridDim.x * blockDim.x) {
        const long long x = r % nx, y = r / nx;
        slot[hilbert_d(n, x, y)] = (int32_t)r;
    }
}

__global__ void k_fill_i32(int32_t* p, long long n, int32_t v) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x)
        p[i] = v;
}

// Stable compaction of the occupied slots in key order, one block of 1024
// threads: perm[a] = receiver with the a-th smallest key.
__global__ void __launch_bounds__(1024) k_hilbert_compact(const int32_t* slot, long long nslot, int32_t* perm) {
    __shared__ long long cnt[1024];
    const int t = threadIdx.x;
    const long long per = (nslot + 1023) / 1024;
    const long long lo = t * per, hi = min(nslot, lo + per);
    long long c = 0;
    for (long long i = lo; i < hi; ++i) c += (slot[i] >= 0);
    cnt[t] = c;
    __syncthreads();
    // inclusive Hillis-Steele scan
    for (int off = 1; off < 1024; off <<= 1) {
        long long v = (t >= off) ? cnt[t - off] : 0;
        __syncthreads();
        cnt[t] += v;
        __syncthreads();
    }
    long long pos = cnt[t] - c;
    for (long long i = lo; i < hi; ++i)
        if (slot[i] >= 0) perm[pos++] = slot[i];
}

cudaError_t hilbert_perm(int nx, int ny, int32_t* perm, int32_t* slot, cudaStream_t st) {
    long long n = 1;
    while (n < nx || n < ny) n <<= 1;
    const long long nslot = n * n;
    k_fill_i32<<<256, 256, 0, st>>>(slot, nslot, -1);
    counted(1);
    k_hilbert_scatter<<<256, 256, 0, st>>>(nx, ny, n, slot);
    counted(1);
    k_hilbert_compact<<<1, 1024, 0, st>>>(slot, nslot, perm);
    counted(1);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// alpha = max |D| : per-block maxima of re^2 + im^2 in FP64, then one block.
// ---------------------------------------------------------------------------
// An FP64 square per entry takes FP64 time (46 us for 34 MB; 2 lanes per cycle and
// SM), so a warp squares its 32 entries in FP64 only if an FP32 square among them
// comes within 2^-21 of the largest the warp has met (a margin above the rounding of
// both): every entry that could be the maximum is, the result is the same double,
// and of m such groups about ln m are.  NaN entries are passed over and an Inf
// gives Inf, as the FP64 comparison does.
__global__ void __launch_bounds__(256) k_max_abs2_part(const cf* __restrict__ D, long long n, double* part) {
    double m = 0.0;
    float mf = 0.f;   // the warp's largest FP32 square, less the margin
    auto take = [&](float x, float y) {
        const float f = fmaf(x, x, y * y);
        // not below the margin, or possibly an underflow
        if (!__any_sync(0xffffffffu, f >= mf && f > 0.f || (f < 1e-30f && mf < 1e-29f && (x != 0.f || y != 0.f)))) return;
        const double a = (double)x * x + (double)y * y;
        m = a > m ? a : m;
        // near overflow all of them go to FP64
        const float g = f < 1e38f ? f * (1.f - 4.8e-7f) : 0.f;
        mf = fmaxf(mf, __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(g))));
    };
    const long long stride = (long long)gridDim.x * blockDim.x, i0 = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    const bool vec = (reinterpret_cast<uintptr_t>(D) & 15) == 0;
    const long long n4 = vec ? n >> 1 : 0;
    const float4* D4 = reinterpret_cast<const float4*>(D);
    const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
    for (long long i = i0; i - i0 < n4; i += 4 * stride) {   // the same trips for every lane
        float4 v[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) v[j] = i + j * stride < n4 ? D4[i + j * stride] : z;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            take(v[j].x, v[j].y);
            take(v[j].z, v[j].w);
        }
    }
    for (long long i = 2 * n4 + i0; i - i0 < n; i += stride) {   // what the pairs leave (all of it when D is not 16-byte aligned)
        const cf v = i < n ? D[i] : make_float2(0.f, 0.f);
        take(v.x, v.y);
    }
    __shared__ double sh[256];
    sh[threadIdx.x] = m;
    __syncthreads();
    for (int s = blockDim.x / 2; s > 0; s >>= 1) {
        if (threadIdx.x < s) sh[threadIdx.x] = fmax(sh[threadIdx.x], sh[threadIdx.x + s]);
        __syncthreads();
    }
    if (threadIdx.x == 0) part[blockIdx.x] = sh[0];
}

__global__ void k_max_final_sqrt(const double* part, int nblk, double* out) {
    __shared__ double sh[256];
    double m = 0.0;
    for (int i = threadIdx.x; i < nblk; i += blockDim.x) m = fmax(m, part[i]);
    sh[threadIdx.x] = m;
    __syncthreads();
    for (int s = blockDim.x / 2; s > 0; s >>= 1) {
        if (threadIdx.x < s) sh[threadIdx.x] = fmax(sh[threadIdx.x], sh[threadIdx.x + s]);
        __syncthreads();
    }
    if (threadIdx.x == 0) out[0] = sqrt(sh[0]);
}

cudaError_t max_abs2(const cf* D, long long n, double* part, int nblk, double* out, cudaStream_t st) {
    k_max_abs2_part<<<nblk, 256, 0, st>>>(D, n, part);
    counted(1);
    k_max_final_sqrt<<<1, 256, 0, st>>>(part, nblk, out);
    counted(1);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Dt[a, s] = RN32(D[s, perm[a]] / RN32(alpha)).  Walks D in natural receiver order so both
// the read (a row segment of D) and the write (a row segment of Dt, at row
// inv[r]) are 256-byte contiguous; a 32 x 32 tile is transposed in shared memory.
// ---------------------------------------------------------------------------
__global__ void k_inverse_perm(const int32_t* perm, long long n, int32_t* inv) {
    for (long long a = blockIdx.x * (long long)blockDim.x + threadIdx.x; a < n;
         a += (long long)gridDim.x * blockDim.x)
        inv[perm[a]] = (int32_t)a;
}

__global__ void __launch_bounds__(256) k_permute_normalise(const cf* __restrict__ D, long long ns, long long nr,
                                                            const int32_t* __restrict__ inv,
                                                            const double* __restrict__ alpha_dev,
                                                            cf* __restrict__ Dt) {
    __shared__ cf tile[32][33];
    const long long r0 = (long long)blockIdx.x * 32, s0 = (long long)blockIdx.y * 32;
    const int tx = threadIdx.x, ty = threadIdx.y;  // 32 x 8
    // one IEEE FP32 division by alpha rounded to FP32: Dt = RN(D / RN(alpha))
    const float alpha = (float)alpha_dev[0];
#pragma unroll
    for (int j = 0; j < 32; j += 8) {
        const long long s = s0 + ty + j, r = r0 + tx;
        cf v = make_float2(0.f, 0.f);
        if (s < ns && r < nr) v = D[s * nr + r];
        tile[ty + j][tx] = v;
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < 32; j += 8) {
        const long long r = r0 + ty + j, s = s0 + tx;
        if (r < nr && s < ns) {
            const cf v = tile[tx][ty + j];
            cf o;
            o.x = __fdiv_rn(v.x, alpha);
            o.y = __fdiv_rn(v.y, alpha);
            Dt[(long long)inv[r] * ns + s] = o;
        }
    }
}

cudaError_t permute_normalise(const cf* D, long long ns, long long nr, const int32_t* perm,
                              const double* alpha_dev, cf* Dt, cudaStream_t st) {
    // The perm buffer holds 2*nr slots: perm[0..nr) then its inverse.
    int32_t* inv = const_cast<int32_t*>(perm) + nr;
    k_inverse_perm<<<(unsigned)((nr + 255) / 256), 256, 0, st>>>(perm, nr, inv);
    counted(1);
    dim3 grid((unsigned)((nr + 31) / 32), (unsigned)((ns + 31) / 32));
    k_permute_normalise<<<grid, dim3(32, 8), 0, st>>>(D, ns, nr, inv, alpha_dev, Dt);
    counted(1);
    return cudaGetLastError();
}

// Block of row r: r / b for equal tiles, else the largest i with roff[i] <= r.
__device__ __forceinline__ int block_of(long long r, long long b, const long long* roff, int N) {
    if (!roff) return (int)(r / b);
    int lo = 0, hi = N - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (roff[mid] <= r)
            lo = mid;
        else
            hi = mid - 1;
    }
    return lo;
}

// X_h = C(theta) assembled from the stacked unknown (eq. 6-9, 15).  A block of 256
// threads takes 64 x 64 entries of one tile (r, c), 4 x 4 per thread, with the
// factors' rows staged 32 columns at a time (an entry at a time read 2 k values
// from L1 per entry: 782 us at nr = 4096, rank 26; about 70 us now).  In the reciprocal
// form the mirror entry is written with it, so the result is bitwise symmetric, as
// X_ji = X_ij^T demands; a low-rank diagonal tile evaluates its upper triangle.
// General form (general != 0): the tiles are listed row-major (i N + j) and every
// tile is its own L R^T (or Z).  The sum over the rank runs in order, one fused
// multiply-add after the other.  roff == nullptr: N tiles of size b; else block i
// covers rows roff[i] .. roff[i + 1] - 1.
constexpr int AS_T = 64, AS_K = 32;
__global__ void __launch_bounds__(256) k_assemble(const cf* __restrict__ th, long long nr, long long b, int N,
                                                  const AsmTile* __restrict__ t, cf* __restrict__ Xh, int general,
                                                  const long long* __restrict__ roff, int sub, int t0) {
    // blockIdx.x: sub-block of the tile (sub x sub of them), blockIdx.y: the tile
    int i, j;
    const int e = t0 + blockIdx.y;
    if (general) {
        i = e / N;
        j = e - i * N;
    } else if (e < N) {
        i = j = e;
    } else {   // pair p = e - N: column j is the last with j N - j (j + 1) / 2 <= p
        const int p = e - N;
        int lo = 0, hi = N - 2;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if ((long long)mid * N - (long long)mid * (mid + 1) / 2 <= p)
                lo = mid;
            else
                hi = mid - 1;
        }
        j = lo;
        i = p - (j * N - j * (j + 1) / 2) + j + 1;
    }
    const AsmTile a = t[e];
    const long long ri = roff ? roff[i] : i * b, rj = roff ? roff[j] : j * b;
    const int di = (int)((roff ? roff[i + 1] : ri + b) - ri), dj = (int)((roff ? roff[j + 1] : rj + b) - rj);
    const int r0 = blockIdx.x / sub * AS_T, c0 = blockIdx.x % sub * AS_T;
    if (r0 >= di || c0 >= dj) return;
    const bool diag = i == j && !general;
    if (diag && r0 > c0) return;   // written as a mirror
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    float2 acc[4][4];
    // the factors' rows (two of 64 x 33), then the mirrored block (64 x 65)
    __shared__ cf buf[2 * AS_T * (AS_K + 1)];
    static_assert(2 * (AS_K + 1) >= AS_T + 1, "the mirrored block fits");
    if (i == j && a.dense) {
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
            for (int v = 0; v < 4; ++v) {
                const int r = r0 + ty + 16 * u, c = c0 + tx + 16 * v;
                acc[u][v] = make_float2(0.f, 0.f);
                if (r >= di || c >= dj) continue;
                const cf x = th[a.off_l + (long long)r * di + c];
                acc[u][v] = x;
                if (diag) {
                    const cf y = th[a.off_l + (long long)c * di + r];
                    acc[u][v] = make_float2(0.5f * (x.x + y.x), 0.5f * (x.y + y.y));
                }
            }
    } else {
        cf(*Ls)[AS_K + 1] = reinterpret_cast<cf(*)[AS_K + 1]>(buf);
        cf(*Rs)[AS_K + 1] = Ls + AS_T;
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
            for (int v = 0; v < 4; ++v) acc[u][v] = make_float2(0.f, 0.f);
        for (int k0 = 0; k0 < a.k; k0 += AS_K) {
            const int kn = min(AS_K, a.k - k0);
            __syncthreads();
            for (int q = threadIdx.x; q < AS_T * AS_K; q += 256) {
                const int r = q / AS_K, k = q % AS_K;
                const bool in = k < kn;
                Ls[r][k] = in && r0 + r < di ? th[a.off_l + (long long)(r0 + r) * a.k + k0 + k] : make_float2(0.f, 0.f);
                Rs[r][k] = in && c0 + r < dj ? th[a.off_r + (long long)(c0 + r) * a.k + k0 + k] : make_float2(0.f, 0.f);
            }
            __syncthreads();
            for (int k = 0; k < kn; ++k) {
                cf l[4], m[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) l[u] = Ls[ty + 16 * u][k];
#pragma unroll
                for (int v = 0; v < 4; ++v) m[v] = Rs[tx + 16 * v][k];
#pragma unroll
                for (int u = 0; u < 4; ++u)
#pragma unroll
                    for (int v = 0; v < 4; ++v) {
                        acc[u][v].x = fmaf(l[u].x, m[v].x, fmaf(-l[u].y, m[v].y, acc[u][v].x));
                        acc[u][v].y = fmaf(l[u].x, m[v].y, fmaf(l[u].y, m[v].x, acc[u][v].y));
                    }
            }
        }
    }
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            const int r = r0 + ty + 16 * u, c = c0 + tx + 16 * v;
            if (r < di && c < dj && !(diag && r > c)) Xh[(ri + r) * nr + rj + c] = acc[u][v];
        }
    if (general) return;
    // the mirror, through shared memory so that its rows are written whole
    cf(*M)[AS_T + 1] = reinterpret_cast<cf(*)[AS_T + 1]>(buf);
    __syncthreads();
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int v = 0; v < 4; ++v) M[tx + 16 * v][ty + 16 * u] = acc[u][v];
    __syncthreads();
    for (int q = threadIdx.x; q < AS_T * AS_T; q += 256) {
        const int c = q / AS_T, r = q % AS_T;   // entry (r0 + r, c0 + c) to (c0 + c, r0 + r)
        if (r0 + r < di && c0 + c < dj && !(diag && r0 + r >= c0 + c)) Xh[(rj + c0 + c) * nr + ri + r0 + r] = M[c][r];
    }
}

cudaError_t assemble_dense(const cf* theta, long long nr, long long b, int N, const AsmTile* tiles, cf* Xh,
                           cudaStream_t st, int general, const long long* roff) {
    const int sub = (int)((b + AS_T - 1) / AS_T);   // b: the largest tile
    const long long nt = general ? (long long)N * N : (long long)N * (N + 1) / 2;
    for (long long t0 = 0; t0 < nt; t0 += 65535) {
        const unsigned cnt = (unsigned)std::min<long long>(65535, nt - t0);
        k_assemble<<<dim3((unsigned)(sub * sub), cnt), 256, 0, st>>>(theta, nr, b, N, tiles, Xh, general, roff, sub,
                                                                     (int)t0);
        counted(1);
    }
    return cudaGetLastError();
}

// X[r, q] = Xh[inv[r], inv[q]]  (X = S X_h S^T): rows of X whole, the gather along
// a row of X_h that fits L1
__global__ void __launch_bounds__(256) k_unpermute(const cf* __restrict__ Xh, long long nr,
                                                   const int32_t* __restrict__ inv, cf* __restrict__ X) {
    for (long long r = blockIdx.x; r < nr; r += gridDim.x) {
        const cf* src = Xh + (long long)inv[r] * nr;
        cf* dst = X + r * nr;
#pragma unroll 4
        for (long long q = threadIdx.x; q < nr; q += blockDim.x) dst[q] = src[inv[q]];
    }
}

cudaError_t unpermute_dense(const cf* Xh, long long nr, const int32_t* perm, cf* X, cudaStream_t st) {
    const int32_t* inv = perm + nr;
    k_unpermute<<<(unsigned)std::min<long long>(nr, 152 * 16), 256, 0, st>>>(Xh, nr, inv, X);
    counted(1);
    return cudaGetLastError();
}

}  // namespace tlr
