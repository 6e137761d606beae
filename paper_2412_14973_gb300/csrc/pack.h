// The packed tile formats of the tensor-core operands (described at the top of
// k_gemm_tcp.cu): a row's 8 values of one k-group, stored and loaded.
#pragma once

#include <cuda_bf16.h>

#include "internal.h"

namespace tlr {

constexpr int kPackTile = 16384;   // bytes of one packed 128 x 16 tile (both formats)

// byte offset of row r's first 16-byte group (k 0 .. 7 for BF16, k 0 .. 3
// for TF32) inside a packed tile's first plane
__device__ __forceinline__ int row_off(int fmt, int r) {
    return (r >> 3) * (fmt == kFmtTF32 ? 512 : 256) + (r & 7) * 16;
}

// TF32 bit pattern of x rounded to nearest, ties away from zero
__device__ __forceinline__ uint32_t tf32_rna(float x) {
    uint32_t r;
    asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
    return r;
}

// The 8 complex values of k-group kg (k = 8 kg .. 8 kg + 7) of one row of a
// packed tile, row = tile + row_off(fmt, r); the imaginary parts times sgn.
__device__ __forceinline__ void pk_store8(char* row, int fmt, int kg, const float2* v, float sgn) {
    if (fmt == kFmtTF32) {
        uint32_t re[8], im[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            re[j] = tf32_rna(v[j].x);
            im[j] = tf32_rna(v[j].y * sgn);
        }
        char* p = row + kg * 256;
        *reinterpret_cast<uint4*>(p) = make_uint4(re[0], re[1], re[2], re[3]);
        *reinterpret_cast<uint4*>(p + 128) = make_uint4(re[4], re[5], re[6], re[7]);
        *reinterpret_cast<uint4*>(p + 8192) = make_uint4(im[0], im[1], im[2], im[3]);
        *reinterpret_cast<uint4*>(p + 8192 + 128) = make_uint4(im[4], im[5], im[6], im[7]);
        return;
    }
    uint32_t w[4][4];
#pragma unroll
    for (int j = 0; j < 8; j += 2) {
        const float x[2][2] = {{v[j].x, v[j + 1].x}, {v[j].y * sgn, v[j + 1].y * sgn}};
#pragma unroll
        for (int p = 0; p < 2; ++p) {
            const __nv_bfloat162 hi = __floats2bfloat162_rn(x[p][0], x[p][1]);
            const float2 hf = __bfloat1622float2(hi);
            const __nv_bfloat162 lo = __floats2bfloat162_rn(x[p][0] - hf.x, x[p][1] - hf.y);
            w[2 * p][j >> 1] = *reinterpret_cast<const uint32_t*>(&hi);
            w[2 * p + 1][j >> 1] = *reinterpret_cast<const uint32_t*>(&lo);
        }
    }
    char* dst = row + kg * 128;
#pragma unroll
    for (int q = 0; q < 4; ++q)
        *reinterpret_cast<uint4*>(dst + q * 4096) = make_uint4(w[q][0], w[q][1], w[q][2], w[q][3]);
}

// Two neighbouring values, k = 2 q and 2 q + 1 (q < 8) of a row of a packed tile, row
// as for pk_store8: 4 bytes per plane (BF16x3) or 8 (TF32)
__device__ __forceinline__ void pk_store2(char* row, int fmt, int q, float2 a, float2 b) {
    if (fmt == kFmtTF32) {
        char* d = row + (q >> 1) * 128 + (q & 1) * 8;
        *reinterpret_cast<uint2*>(d) = make_uint2(tf32_rna(a.x), tf32_rna(b.x));
        *reinterpret_cast<uint2*>(d + 8192) = make_uint2(tf32_rna(a.y), tf32_rna(b.y));
        return;
    }
    char* dst = row + (q >> 2) * 128 + (q & 3) * 4;
    const float x[2][2] = {{a.x, b.x}, {a.y, b.y}};
#pragma unroll
    for (int p = 0; p < 2; ++p) {
        const __nv_bfloat162 hi = __floats2bfloat162_rn(x[p][0], x[p][1]);
        const float2 hf = __bfloat1622float2(hi);
        const __nv_bfloat162 lo = __floats2bfloat162_rn(x[p][0] - hf.x, x[p][1] - hf.y);
        *reinterpret_cast<__nv_bfloat162*>(dst + 2 * p * 4096) = hi;
        *reinterpret_cast<__nv_bfloat162*>(dst + (2 * p + 1) * 4096) = lo;
    }
}

// The inverse: the 8 complex values of k-group kg of a packed row (BF16:
// hi + lo of each part, the BF16 halves widened by moving their bits into the
// high half of an FP32 word; TF32: the stored words).
__device__ __forceinline__ void pk_load8(const char* row, int fmt, int kg, float2* v) {
    if (fmt == kFmtTF32) {
        const char* p = row + kg * 256;
        const uint4 r0 = *reinterpret_cast<const uint4*>(p), r1 = *reinterpret_cast<const uint4*>(p + 128);
        const uint4 i0 = *reinterpret_cast<const uint4*>(p + 8192),
                    i1 = *reinterpret_cast<const uint4*>(p + 8192 + 128);
        const uint32_t re[8] = {r0.x, r0.y, r0.z, r0.w, r1.x, r1.y, r1.z, r1.w};
        const uint32_t im[8] = {i0.x, i0.y, i0.z, i0.w, i1.x, i1.y, i1.z, i1.w};
#pragma unroll
        for (int j = 0; j < 8; ++j) v[j] = make_float2(__uint_as_float(re[j]), __uint_as_float(im[j]));
        return;
    }
    const char* src = row + kg * 128;
    uint4 w[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) w[q] = *reinterpret_cast<const uint4*>(src + q * 4096);
    const uint32_t* wr = reinterpret_cast<const uint32_t*>(&w[0]);
    const uint32_t* wl = reinterpret_cast<const uint32_t*>(&w[1]);
    const uint32_t* wi = reinterpret_cast<const uint32_t*>(&w[2]);
    const uint32_t* wm = reinterpret_cast<const uint32_t*>(&w[3]);
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        const uint32_t sh = (j & 1) * 16;
        v[j] = make_float2(__uint_as_float(((wr[j >> 1] >> sh) & 0xffffu) << 16) +
                               __uint_as_float(((wl[j >> 1] >> sh) & 0xffffu) << 16),
                           __uint_as_float(((wi[j >> 1] >> sh) & 0xffffu) << 16) +
                               __uint_as_float(((wm[j >> 1] >> sh) & 0xffffu) << 16));
    }
}

// Block of the 16-row residual tile starting at row r0: r0 / b for equal
// tiles, else the largest i with roff[i] <= r0 (every roff[i] is a multiple
// of kFuseRows, so the tile lies in it); rl0 = its first row in the block, bK =
// the block's size.
struct RTile {
    int blk, rl0, bK;
};
__device__ __forceinline__ RTile rtile(int r0, int b, const long long* roff, int nblk) {
    RTile t;
    if (roff) {
        int lo = 0, hi = nblk - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (roff[mid] <= r0)
                lo = mid;
            else
                hi = mid - 1;
        }
        t.blk = lo;
        t.rl0 = r0 - (int)roff[lo];
        t.bK = (int)(roff[lo + 1] - roff[lo]);
    } else {
        t.blk = r0 / b;
        t.rl0 = r0 - t.blk * b;
        t.bK = b;
    }
    return t;
}

}  // namespace tlr
