// FP32 grouped complex GEMM on the tensor cores (tcgen05, sm_103a): the
// default-precision path of the TLR contractions -- compress T = F^T Dfrak,
// expand Y = F T~ (+ P Z Dfrak), the factor-gradient projections (eq. 25-27)
// and the dense adjoint G = V Dfrak^H, on FP32 operands in place.
//
// Arithmetic.  Every FP32 value from 2^-109 up is split exactly into three BF16 values
// x = h + m + l (h = RN(x), m = RN(x - h), l = x - h - m: 8 + 8 + 8 significant
// bits), and every real product takes the six of the nine BF16 products that
// are not below 2^-24 of it: hh, hm, mh, hl, mm, lh.  A complex product is four
// real ones (4M), so a 16-deep chunk of a 128 x 128 tile takes 24 MMAs.
// The tensor core adds into its FP32 accumulator without rounding to nearest
// (about half an ulp toward zero per MMA), so the accumulator never carries
// more than one chunk: the smallest products are issued first (while the
// accumulator is still small) and every 16-deep chunk is drained and added to
// FP32 registers, rounding to nearest.  Measured against 64 bits this is below the
// error of FP32 fused multiply-adds over the whole contraction from 13 products on,
// also for same-signed terms, whose signed mean it leaves at -4 to -6e-8 (see
// tests/test_gpu_gemm_f32.py, test_gpu_gemm_f32_range.py).
//
// What bounds it: the workers' split and drain (issue slots 60 % used, tensor pipe 46 %
// active on a dense adjoint of 2048); 24 BF16 products per complex multiply-add of
// 16-deep chunks, 8/48 of the BF16 peak, would be 316 TFLOP/s.  Both run beside the
// MMAs: three warps copy chunks from global memory into a raw shared-memory ring
// (cp.async, gather applied, zeros from the k tail on), 16 worker warps split
// chunk c into the tensor core's canonical K-major no-swizzle layout (8-row x
// 16-byte core matrices) and drain chunk c - 2 from one of two TMEM accumulator
// pairs, while the tensor core works on chunk c - 1 and another warp issues chunk
// c's MMAs.  The split takes fewer issue slots than the SM has under 24 MMAs (it
// bounded the 12-MMA form), so no operand is packed in memory and the kernel
// needs no workspace.  The roles are apart because a worker's 64 accumulators
// leave no registers for cursors, and beside this much shared memory the L1
// holds no spills.  Tried on nr = ns = 4096 (dense adjoint, TFLOP/s; the MMAs
// alone: 285): copies and cursors in the workers 58 to 83 (spills) and 176, the
// MMAs issued by a worker 125, one copy warp per operand 191 to 204 (65 cycles
// per copy instruction), bulk copies of 128 bytes 74 (31 cycles each); this form
// 225, with the checks below 215 (the FP32 FMA kernel before: 34).
// Persistent: one CTA per SM walks the output tiles, its pipeline running
// across tile ends.
//
// Values beyond the split: Inf, NaN or a magnitude that rounds to Inf in BF16 make a
// tile's results non-finite; a value other than zero below 2^-109 has a third part
// below BF16's smallest and is found while it is split.  What they touch is computed
// again with plain FP32 fused multiply-adds (plain_tile): the non-finite results, results
// below 2^-100, or the whole tile.  So Inf, NaN and small values come out as FP32
// arithmetic gives them, at 13 TFLOP/s (all of nr = ns = 4096 42 ms, a NaN row 11 ms).
//
// Every barrier wait is bounded (2 s); a timeout is recorded in the error word.
#include <cuda_bf16.h>

#include <algorithm>

#include "internal.h"

namespace tlr {

namespace {

constexpr int TM = 128, TN = 128, KC = 16;
constexpr int NW = 16;                              // worker warps
constexpr int WMMA = NW, WCOPY = NW + 1, NCOPY = 3; // the MMA warp, the copy warps
constexpr int NTHR = (NW + 4) * 32;                 // whole warps per scheduler
constexpr int PLANE = 128 * KC * 2;                 // one BF16 plane of a 128 x 16 operand tile
constexpr int TILE = 6 * PLANE;                     // Re h, m, l, Im h, m, l
constexpr int STAGE = 2 * TILE;                     // A and B
constexpr int NSTAGE = 3;
constexpr int LAG = 2;                              // chunks between split and drain
constexpr int RAW_OP = 128 * KC * 8;                // one operand's raw chunk: 128 rows x 128 B, or 16 k x 1 KB
constexpr int NRAW = 2;
constexpr int RAW_OFF = NSTAGE * STAGE;
constexpr int ROW_OFF = RAW_OFF + NRAW * 2 * RAW_OP;   // per copy warp: element offsets of A's and B's 128 rows
constexpr int CTRL_OFF = ROW_OFF + NCOPY * 2 * 128 * 8;
constexpr int SMEM_BYTES = CTRL_OFF + 256;
constexpr uint32_t TMEM_COLS = 512;                 // two pairs of 2 x 128 columns
constexpr unsigned long long WAIT_NS = 2000000000ull;
static_assert(SMEM_BYTES <= 227 * 1024, "shared memory budget");

// instruction descriptor: FP32 accumulator, BF16 x BF16, M 128; N / 8 goes to bits 17-22
constexpr uint32_t IDESC = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(TM >> 4) << 24);
constexpr uint32_t NEG_A = 1u << 13;

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// shared-memory matrix descriptor, K-major no-swizzle: core matrices 128 B
// apart along K and 256 B apart along rows
__device__ __forceinline__ uint64_t sdesc(uint32_t saddr) {
    return (uint64_t)((saddr >> 4) & 0x3FFFu) | ((uint64_t)(128u >> 4) << 16) | ((uint64_t)(256u >> 4) << 32) |
           ((uint64_t)1 << 46);
}

__device__ __forceinline__ unsigned long long now_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, const volatile int* abort_flag) {
    unsigned long long t0 = 0;
    for (unsigned it = 0;; ++it) {
        uint32_t ok;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(ok)
            : "r"(bar), "r"(parity)
            : "memory");
        if (ok) return true;
        if ((it & 255u) == 255u) {
            if (*abort_flag) return false;
            const unsigned long long t = now_ns();
            if (t0 == 0)
                t0 = t;
            else if (t - t0 > WAIT_NS)
                return false;
        }
    }
}

__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

__device__ __forceinline__ void commit(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}

__device__ __forceinline__ void mma(uint32_t tmem, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        :
        : "r"(tmem), "l"(a), "l"(b), "r"(idesc), "r"(acc)
        : "memory");
}

__device__ __forceinline__ void tmem_ld16(uint32_t addr, uint32_t* r) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(addr));
}

// two FP32 operations per instruction
__device__ __forceinline__ uint64_t pair(float lo, float hi) {
    return ((uint64_t)__float_as_uint(hi) << 32) | __float_as_uint(lo);
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
    uint64_t r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}

// most = max(most, |x0|, |x1|), NaN if any is
__device__ __forceinline__ void max_abs(float& most, float x0, float x1) {
    asm("max.NaN.abs.f32 %0, %0, %1, %2;" : "+f"(most) : "f"(x0), "f"(x1));
}

// a magnitude's bits, doubled, less one: zero becomes the largest
__device__ __forceinline__ uint32_t twice(float x) { return 2u * __float_as_uint(x) - 1u; }

// h, m, l of two FP32 values as BF16 pairs (x0 in the low half); least: the smallest
// twice() so far
__device__ __forceinline__ void split2(float x0, float x1, uint32_t* w, uint32_t& least) {
    least = __vimin3_u32(least, twice(x0), twice(x1));
    uint64_t x = pair(x0, x1);
#pragma unroll
    for (int p = 0; p < 3; ++p) {
        const __nv_bfloat162 b = __floats2bfloat162_rn(__uint_as_float((uint32_t)x), __uint_as_float((uint32_t)(x >> 32)));
        const uint32_t u = *reinterpret_cast<const uint32_t*>(&b);
        w[p] = u;
        // minus the BF16 values (their sign bits flipped)
        if (p < 2)
            x = add2(x, ((uint64_t)((u & 0xffff0000u) ^ 0x80000000u) << 32) | ((u << 16) ^ 0x80000000u));
    }
}

// ---------------------------------------------------------------------------
// work items: (M tile fastest, N tile, problem and split)
// ---------------------------------------------------------------------------
struct Item {
    const GProb* P;
    int m0, n0, chunk;
};

struct Launch {
    const GProb* probs;
    int nsplit, kchunk, nx, ny;
    int nitems;         // below 2^31 - grid (gemm_f32)
    int epi;
    int shallow;        // 0: no item has 1 .. SHALLOW products per output
    long long part_stride;
};

__device__ __forceinline__ bool item_at(const Launch& L, int i, Item& it) {
    const int xy = L.nx * L.ny;
    const int z = i / xy, r = i - z * xy;
    const int prob = z / L.nsplit;
    it.chunk = z - prob * L.nsplit;
    it.m0 = (r % L.ny) * TM;
    it.n0 = (r / L.ny) * TN;
    it.P = L.probs + prob;
    return it.m0 < it.P->M && it.n0 < it.P->N;
}

// the K range [kb, ke) of a term (kb a multiple of 16)
__device__ __forceinline__ void k_range(const Launch& L, const Item& it, int K, int& kb, int& ke) {
    kb = 0;
    ke = K;
    if (L.nsplit > 1) {
        kb = it.chunk * L.kchunk;
        ke = min(K, kb + L.kchunk);
    }
}

// An item's products per output: up to SHALLOW of them are left to plain FP32
// multiply-adds (plain_tile), which round less often than the drained chunk's 24 MMAs
// do: 1 product 3.0e-8 against 4.7e-8, 8 same-signed ones 4.6e-8 against 4.8e-8, 16
// already 6.1e-8 against 4.6e-8 (relative error in norm).
constexpr int SHALLOW = kF32Shallow;
__device__ __forceinline__ int depth_of(const Launch& L, const Item& it) {
    int d = 0;
    for (int t = 0; t < it.P->nt; ++t) {
        int kb, ke;
        k_range(L, it, it.P->t[t].K, kb, ke);
        d += max(0, ke - kb);
    }
    return d;
}

// the chunks that an item gives the tensor cores
__device__ __forceinline__ int chunks_of(const Launch& L, const Item& it) {
    if (L.shallow && depth_of(L, it) <= SHALLOW) return 0;
    int C = 0;
    for (int t = 0; t < it.P->nt; ++t) {
        int kb, ke;
        k_range(L, it, it.P->t[t].K, kb, ke);
        if (ke > kb) C += (ke - kb + KC - 1) / KC;
    }
    return C;
}

// ---------------------------------------------------------------------------
// copying and splitting one operand's 16-deep chunk
// ---------------------------------------------------------------------------

__device__ __forceinline__ void copy16(uint32_t dst, const void* src, int bytes) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void copy8(uint32_t dst, const void* src, bool in) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(dst), "l"(src), "r"(in ? 8 : 0) : "memory");
}

// one operand of one term as a copy warp sees it
struct Opnd {
    const cf* base;      // k contiguous: row r at base + rowoff[r]; rows contiguous: base + k ld (k through g)
    const int* g;
    const long long* rowoff;
    long long ld;
    int rows;            // valid rows of the tile
    bool vec;            // every row piece starts on 16 bytes
};

template <bool KCONTIG>
__device__ __forceinline__ Opnd make_opnd(const cf* base, long long ld, const int* g, int R, int r0,
                                          long long* rowoff, int lane) {
    Opnd o;
    o.g = g;
    o.ld = ld;
    o.rows = min(128, R - r0);
    o.rowoff = rowoff;
    o.vec = (ld & 1) == 0;
    if (KCONTIG) {
        __syncwarp();
        for (int r = lane; r < o.rows; r += 32) rowoff[r] = (long long)(g ? g[r0 + r] : r0 + r) * ld;
        __syncwarp();
    } else {
        base += r0;
        o.vec = o.vec && (o.rows & 1) == 0;
    }
    o.base = base;
    o.vec = o.vec && (reinterpret_cast<uintptr_t>(base) & 15) == 0;
    return o;
}

// raw position of 16-byte column q (two k) of row r, k contiguous: columns
// rotated by the row so that 8 rows of one column lie in 8 different ones
__device__ __forceinline__ int raw_pos(int r, int q) { return r * 128 + ((q ^ (r & 7)) << 4); }

// Copy warp w of NCOPY starts its copies of chunk k0 .. k0 + 15, zeros from ke on.
// Rows beyond the operand keep what the ring held: they reach only results that
// are not stored.  k contiguous: 8 lanes take a row's 128 bytes; rows contiguous:
// 512 bytes of one k per instruction.
template <bool KCONTIG>
__device__ __forceinline__ void copy_chunk(const Opnd& o, int k0, int ke, int w, uint32_t raw, int lane) {
    if (KCONTIG) {
        if (o.vec) {
            const int q = lane & 7, n = max(0, min(2, ke - k0 - 2 * q)) * 8;   // bytes
            const cf* p = n ? o.base + k0 + 2 * q : o.base;
#pragma unroll
            for (int i = 0; i < 11; ++i) {
                const int r = (i * NCOPY + w) * 4 + (lane >> 3);
                if (r < o.rows) copy16(raw + raw_pos(r, q), p + o.rowoff[r], n);
            }
        } else {
            const int q = lane & 15;
            const bool in = k0 + q < ke;
            const cf* p = o.base + (in ? k0 + q : 0);
#pragma unroll 4
            for (int i = w; i < 64; i += NCOPY) {
                const int r = i * 2 + (lane >> 4);
                if (r < o.rows) copy8(raw + raw_pos(r, q >> 1) + (q & 1) * 8, p + o.rowoff[r], in);
            }
        }
    } else {
        const int k = k0 + (lane & 15);
        const int gi = k < ke ? (o.g ? o.g[k] : k) : -1;
#pragma unroll
        for (int i = 0; i < 11; ++i) {
            const int e = i * NCOPY + w;   // half (e & 1) of k e >> 1
            const int row = __shfl_sync(0xffffffffu, gi, (e >> 1) & 15);
            const bool in = row >= 0;
            const int r = (e & 1) * 64 + lane * 2;
            if (e < 2 * KC && r < o.rows) {
                const cf* p = in ? o.base + (long long)row * o.ld + r : o.base;
                const uint32_t d = raw + (e >> 1) * 1024 + r * 8;
                if (o.vec) {
                    copy16(d, p, in ? 16 : 0);
                } else {
                    copy8(d, p, in);
                    if (r + 1 < o.rows) copy8(d + 8, in ? p + 1 : o.base, in);
                }
            }
        }
    }
}

// Splits a raw chunk into the operand tile, four k at a time (8 values and 12
// words live beside the 64 accumulators).  Both the reads (8 rows of a phase in
// 8 different columns, or consecutive rows) and the 8-byte stores (rows 8 to 15
// of 16 take the other half of the k-group: together all banks) are free of
// bank conflicts.  k contiguous: thread = (row, half of each k-group); rows
// contiguous: thread = (row, k-group).  True where a value other than zero is below
// 2^-109, so that its split may not be exact (1.5 instructions a value; the smallest
// magnitude by floating-point minima takes half of one, but zeros have to be told apart
// then, which cost more where there are any).
template <bool KCONTIG>
__device__ __forceinline__ bool split_chunk(char* tile, const char* raw, int t8) {
    uint32_t least = ~0u;
    const int r = KCONTIG ? (t8 >> 5) * 16 + (t8 & 15) : t8 & 127;
    const int odd = (r >> 3) & 1;
    char* const d = tile + (r >> 3) * 256 + (r & 7) * 16;
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        float2 v[4];
        const int kg = KCONTIG ? j : t8 >> 7;
        const int h = (KCONTIG ? (t8 >> 4) & 1 : j) ^ odd;   // k 8 kg + 4 h ..
        if (KCONTIG) {
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                const float4 x = *reinterpret_cast<const float4*>(raw + raw_pos(r, kg * 4 + h * 2 + i));
                v[2 * i] = make_float2(x.x, x.y);
                v[2 * i + 1] = make_float2(x.z, x.w);
            }
        } else {
            const char* q = raw + (kg * 8 + h * 4) * 1024 + r * 8;
#pragma unroll
            for (int i = 0; i < 4; ++i) v[i] = *reinterpret_cast<const float2*>(q + i * 1024);
        }
        char* const o = d + kg * 128 + h * 8;
        uint32_t w[2][3];
        split2(v[0].x, v[1].x, w[0], least);
        split2(v[2].x, v[3].x, w[1], least);
#pragma unroll
        for (int p = 0; p < 3; ++p) *reinterpret_cast<uint2*>(o + p * PLANE) = make_uint2(w[0][p], w[1][p]);
        split2(v[0].y, v[1].y, w[0], least);
        split2(v[2].y, v[3].y, w[1], least);
#pragma unroll
        for (int p = 0; p < 3; ++p) *reinterpret_cast<uint2*>(o + (3 + p) * PLANE) = make_uint2(w[0][p], w[1][p]);
    }
    return least < 2u * ((uint32_t)(127 - 109) << 23) - 1u;
}

// A result that the tensor cores gave as plain FP32 multiply-adds would, up to its
// rounding: zero, or from 2^-100 up and finite (below, the sums' own rounding nears
// FP32's smallest values, which the tensor core meets 24 times a chunk).
__device__ __forceinline__ bool good(float x) {
    const uint32_t u = __float_as_uint(x) & 0x7fffffffu, lo = (uint32_t)(127 - 100) << 23;
    return u == 0u || u - lo < 0x7f800000u - lo;
}

// Recomputes results of a warp's 32 x 32 part of a tile just written by plain FP32
// fused multiply-adds along k: all of them, or those that are not good().  The warp
// works on 32 x 16 at a time, a lane on 4 rows (8 apart) and 4 columns (4 apart), so
// an operand row read from L1 or L2 serves 4 products (one lane per row, an output
// after the other, read each operand row for one).
template <int AM, int BMD>
__device__ __forceinline__ void plain_tile(const Launch& L, int item, bool all) {
    const int lane = threadIdx.x & 31, lg = (threadIdx.x >> 5) & 3, cg = threadIdx.x >> 7, epi = L.epi;
    Item it;
    item_at(L, item, it);
    const GProb& P = *it.P;
    const int m0 = it.m0 + lg * 32 + (lane & 7);
    cf* const C = P.C + (epi == EPI_PARTIAL ? it.chunk * L.part_stride : 0);
    __syncwarp();   // the other lanes' results are read below
    for (int half = 0; half < 2; ++half) {
        const int n0 = it.n0 + cg * 32 + half * 16 + (lane >> 3);
        unsigned todo = 0;
#pragma unroll
        for (int e = 0; e < 16; ++e) {
            const int m = m0 + (e >> 2) * 8, n = n0 + (e & 3) * 4;
            if (m < P.M && n < P.N) {
                bool again = all;
                if (!all) {
                    const float2 v = C[(long long)m * P.ldc + n];
                    again = !good(v.x) || !good(v.y);
                }
                if (again) todo |= 1u << e;
            }
        }
        if (!__any_sync(0xffffffffu, todo != 0u)) continue;
        float2 c[16];
#pragma unroll
        for (int e = 0; e < 16; ++e) c[e] = make_float2(0.f, 0.f);
        for (int ti = 0; ti < P.nt; ++ti) {
            const GTerm& t = P.t[ti];
            int kb, ke;
            k_range(L, it, t.K, kb, ke);
            const cf* a[4];
            const cf* b[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {   // rows and columns beyond the operands read the last
                const int m = min(m0 + i * 8, P.M - 1), n = min(n0 + i * 4, P.N - 1);
                a[i] = AM == A_KM ? t.A + m : t.A + (long long)m * t.lda;
                b[i] = BMD == B_KN ? t.B + n : t.B + (long long)(t.g ? t.g[n] : n) * t.ldb;
            }
            const float sa = t.sa, sb = t.sb;
            for (int k = kb; k < ke; ++k) {
                const long long ao = AM == A_KM ? (long long)k * t.lda : k;
                const long long bo = BMD == B_KN ? (long long)(t.g ? t.g[k] : k) * t.ldb : k;
                float2 x[4], y[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    x[i] = a[i][ao];
                    x[i].y *= sa;
                    y[i] = b[i][bo];
                    y[i].y *= sb;
                }
#pragma unroll
                for (int e = 0; e < 16; ++e) {
                    const float2 u = x[e >> 2], v = y[e & 3];
                    c[e].x = fmaf(u.x, v.x, c[e].x);
                    c[e].x = fmaf(-u.y, v.y, c[e].x);
                    c[e].y = fmaf(u.x, v.y, c[e].y);
                    c[e].y = fmaf(u.y, v.x, c[e].y);
                }
            }
        }
#pragma unroll
        for (int e = 0; e < 16; ++e) {
            if (!(todo >> e & 1u)) continue;
            const long long o = (long long)(m0 + (e >> 2) * 8) * P.ldc + n0 + (e & 3) * 4;
            if (epi == EPI_SUB) {
                const float2 s = P.S[o];
                c[e].x -= s.x;
                c[e].y -= s.y;
            }
            C[o] = c[e];
        }
    }
}

// A warp's part of this CTA's items: those without chunks and those with any of the
// chunks span[0] .. span[1] as a whole, of the items span[2] .. span[3] what is not good()
template <int AM, int BMD>
__device__ __noinline__ void plain_items(const Launch& L, const int* span) {
    int c = 0;
    for (int i = blockIdx.x; i < L.nitems; i += gridDim.x) {
        Item it;
        if (!item_at(L, i, it)) continue;
        const int C = chunks_of(L, it);
        const bool all = C == 0 || (c <= span[1] && c + C > span[0]);
        if (all || (i >= span[2] && i <= span[3])) plain_tile<AM, BMD>(L, i, all);
        c += C;
    }
}

// Writes a thread's row of 32 columns (real parts of pairs of columns, then
// imaginary parts) to the tile's destination, 16 bytes at a time; consecutive
// stores fill the row's 32-byte sectors.  (No room for a staging transpose in
// shared memory; the stores run beside the next tile's first MMAs.)  True if
// any value is not good().
__device__ __forceinline__ bool write_tile(const Launch& L, const Item& it, const uint64_t* acc, int lg, int cg,
                                           int lane) {
    const int epi = L.epi;
    const GProb& P = *it.P;
    const int m = it.m0 + lg * 32 + lane, nb = it.n0 + cg * 32, N = P.N;
    if (m >= P.M) return false;
    cf* const Cp = P.C + (epi == EPI_PARTIAL ? it.chunk * L.part_stride : 0) + (long long)m * P.ldc + nb;
    const cf* const Sp = epi == EPI_SUB ? P.S + (long long)m * P.ldc + nb : nullptr;
    const bool vec = ((reinterpret_cast<uintptr_t>(Cp) | reinterpret_cast<uintptr_t>(Sp)) & 15) == 0;
    float most = 0.f;
    uint32_t least = ~0u;
#pragma unroll
    for (int q = 0; q < 16; ++q) {
        if (nb + 2 * q < N) {
            const bool two = nb + 2 * q + 1 < N;
            float4 v = make_float4(__uint_as_float((uint32_t)acc[q]), __uint_as_float((uint32_t)acc[16 + q]),
                                   __uint_as_float((uint32_t)(acc[q] >> 32)),
                                   __uint_as_float((uint32_t)(acc[16 + q] >> 32)));
            if (epi == EPI_SUB) {
                if (vec && two) {
                    const float4 s = *reinterpret_cast<const float4*>(Sp + 2 * q);
                    v.x -= s.x;
                    v.y -= s.y;
                    v.z -= s.z;
                    v.w -= s.w;
                } else {
                    v.x -= Sp[2 * q].x;
                    v.y -= Sp[2 * q].y;
                    if (two) {
                        v.z -= Sp[2 * q + 1].x;
                        v.w -= Sp[2 * q + 1].y;
                    }
                }
            }
            // of a single column twice the same value
            const float z = two ? v.z : v.x, w = two ? v.w : v.y;
            max_abs(most, v.x, v.y);
            max_abs(most, z, w);
            least = __vimin3_u32(least, twice(v.x), twice(v.y));
            least = __vimin3_u32(least, twice(z), twice(w));
            if (vec && two) {
                *reinterpret_cast<float4*>(Cp + 2 * q) = v;
            } else {
                Cp[2 * q] = make_float2(v.x, v.y);
                if (two) Cp[2 * q + 1] = make_float2(v.z, v.w);
            }
        }
    }
    return least < 2u * ((uint32_t)(127 - 100) << 23) - 1u || !(most < INFINITY);
}

template <int AM, int BMD>
__global__ void __launch_bounds__(NTHR, 1) k_cgemm_f32(const __grid_constant__ Launch L, int* err) {
    chain_wait();
    extern __shared__ __align__(1024) char smem[];
    if (*(volatile int*)err != 0) return;   // an earlier contraction gave up: do no more work
    uint64_t* full = reinterpret_cast<uint64_t*>(smem + CTRL_OFF);   // operand stage split (one arrival per worker warp)
    uint64_t* empty = full + NSTAGE;        // operand stage read by its MMAs
    uint64_t* tfull = empty + NSTAGE;       // [2] accumulator pair holds a chunk
    uint64_t* tempty = tfull + 2;           // [2] accumulator pair drained (one arrival per worker warp)
    uint64_t* rfull = tempty + 2;           // [NRAW] raw chunk landed (every copy lane's copies)
    uint64_t* rempty = rfull + NRAW;        // [NRAW] raw chunk read (one arrival per worker warp)
    uint32_t* tslot = reinterpret_cast<uint32_t*>(rempty + NRAW);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tslot + 1);
    // what is computed again: the first and last of this CTA's chunks with a value whose
    // split may not be exact, the first and last item with results that are not good(), any
    int* const again = reinterpret_cast<int*>(tslot + 2);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int s = 0; s < NSTAGE; ++s) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(&full[s])), "r"(NW) : "memory");
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&empty[s])) : "memory");
        }
        for (int b = 0; b < 2; ++b) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&tfull[b])) : "memory");
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(&tempty[b])), "r"(NW) : "memory");
        }
        for (int r = 0; r < NRAW; ++r) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(&rfull[r])), "r"(NCOPY * 32) : "memory");
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(&rempty[r])), "r"(NW) : "memory");
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        *abort_flag = 0;
        again[0] = again[2] = INT_MAX;
        again[1] = again[3] = -1;
        again[4] = again[5] = 0;   // (the last stays zero: a wait that nobody ends early)
    }
    // ones where no copy goes (rows beyond an operand), so that nothing left there by
    // another kernel is taken for a small value
    for (int e = threadIdx.x; e < NRAW * 2 * RAW_OP / 16; e += NTHR)
        reinterpret_cast<float4*>(smem + RAW_OFF)[e] = make_float4(1.f, 1.f, 1.f, 1.f);
    if (warp == WMMA) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tslot)),
                     "r"(TMEM_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = *tslot;

    if (warp == WMMA) {
        if (lane == 0) {
            // ---------------- MMA issuer: one chunk after the other, across tiles ----------------
            int c = 0;
            for (int i = blockIdx.x; i < L.nitems && !*abort_flag; i += gridDim.x) {
                Item it;
                if (!item_at(L, i, it) || (L.shallow && depth_of(L, it) <= SHALLOW)) continue;
                // a ragged last N tile computes only its 16-column groups
                const uint32_t idesc = IDESC | ((uint32_t)(min(TN, (it.P->N - it.n0 + 15) & ~15) >> 3) << 17);
                for (int t = 0; t < it.P->nt && !*abort_flag; ++t) {
                    int k0, ke;
                    k_range(L, it, it.P->t[t].K, k0, ke);
                    // Cr = Ar Br - sa sb Ai Bi, Ci = sb Ar Bi + sa Ai Br (sa, sb: -1 for a conjugated operand)
                    const bool ca = it.P->t[t].sa < 0.f, cb = it.P->t[t].sb < 0.f;
                    const uint32_t id_ii = idesc | (ca == cb ? NEG_A : 0u), id_ri = idesc | (cb ? NEG_A : 0u),
                                   id_ir = idesc | (ca ? NEG_A : 0u);
                    for (; k0 < ke; k0 += KC, ++c) {
                        const int s = c % NSTAGE, b = c & 1;
                        if (!mbar_wait(smem_u32(&full[s]), (uint32_t)((c / NSTAGE) & 1), abort_flag) ||
                            (c >= 2 && !mbar_wait(smem_u32(&tempty[b]), (uint32_t)(((c >> 1) - 1) & 1), abort_flag))) {
                            *abort_flag = 1;
                            break;
                        }
                        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                        const uint32_t a0 = smem_u32(smem + s * STAGE);
                        const uint64_t ar = sdesc(a0), br = sdesc(a0 + TILE);
                        constexpr uint64_t D = PLANE >> 4;   // one plane further (0 h, 1 m, 2 l; + 3: Im)
                        const uint64_t ai = ar + 3 * D, bi = br + 3 * D;
                        const uint32_t dr = tmem + b * 2 * TN, di = dr + TN;
                        // products of the order of 2^-16, then 2^-8, then 1
#pragma unroll
                        for (int order = 2; order >= 0; --order)
#pragma unroll
                            for (int p = 0; p <= order; ++p) {
                                const int q = order - p;
                                mma(dr, ar + p * D, br + q * D, idesc, order == 2 && p == 0 ? 0u : 1u);
                                mma(di, ar + p * D, bi + q * D, id_ri, order == 2 && p == 0 ? 0u : 1u);
                                mma(dr, ai + p * D, bi + q * D, id_ii, 1u);
                                mma(di, ai + p * D, br + q * D, id_ir, 1u);
                            }
                        commit(smem_u32(&empty[s]));
                        commit(smem_u32(&tfull[b]));
                    }
                }
            }
            // after a timeout: the MMAs in flight end (or two seconds pass) before their
            // operands and accumulators are given up
            if (*abort_flag && c > 0)
                (void)mbar_wait(smem_u32(&tfull[(c - 1) & 1]), (uint32_t)(((c - 1) >> 1) & 1), again + 5);
        }
        __syncwarp();
    } else if (warp >= WCOPY) {
        // ---------------- copies, across tiles ----------------
        const int w = warp - WCOPY;
        long long* const rowoff = reinterpret_cast<long long*>(smem + ROW_OFF) + w * 256;
        int c = 0;
        for (int i = blockIdx.x; i < L.nitems && !*abort_flag; i += gridDim.x) {
            Item it;
            if (!item_at(L, i, it) || (L.shallow && depth_of(L, it) <= SHALLOW)) continue;
            for (int t = 0; t < it.P->nt && !*abort_flag; ++t) {
                const GTerm& T = it.P->t[t];
                int k0, ke;
                k_range(L, it, T.K, k0, ke);
                if (k0 >= ke) continue;
                const Opnd oa = make_opnd<AM == A_MK>(T.A, T.lda, nullptr, it.P->M, it.m0, rowoff, lane);
                const Opnd ob = make_opnd<BMD == B_NK>(T.B, T.ldb, T.g, it.P->N, it.n0, rowoff + 128, lane);
                for (; k0 < ke; k0 += KC, ++c) {
                    const int s = c % NRAW;
                    if (c >= NRAW && !mbar_wait(smem_u32(&rempty[s]), (uint32_t)((c / NRAW - 1) & 1), abort_flag)) {
                        *abort_flag = 1;
                        break;
                    }
                    const uint32_t raw = smem_u32(smem + RAW_OFF) + s * 2 * RAW_OP;
                    copy_chunk<AM == A_MK>(oa, k0, ke, w, raw, lane);
                    copy_chunk<BMD == B_NK>(ob, k0, ke, w, raw + RAW_OP, lane);
                    asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(smem_u32(&rfull[s]))
                                 : "memory");
                }
            }
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
    } else if (warp < NW) {
        // ---------------- workers ----------------
        const bool isB = warp >= NW / 2;
        const int t8 = threadIdx.x & 255;
        const int lg = warp & 3, cg = warp >> 2;   // TMEM lanes 32 lg .., columns 32 cg ..
        const uint32_t tm0 = tmem + ((uint32_t)(lg * 32) << 16) + cg * 32;
        // the chunks of this CTA in all (the split runs ahead of the drain, across items)
        int total = 0;
        for (int i = blockIdx.x; i < L.nitems; i += gridDim.x) {
            Item it;
            if (!item_at(L, i, it)) continue;
            const int C = chunks_of(L, it);
            total += C;
            if (C == 0) *(volatile int*)(again + 4) = 1;
        }
        uint64_t acc[32];   // real parts of 32 columns in pairs, then imaginary parts
#pragma unroll
        for (int j = 0; j < 32; ++j) acc[j] = 0;
        // the item whose chunks are being added up, its chunks still to split and to drain
        int ci = (int)blockIdx.x - (int)gridDim.x;
        bool cols = false;   // it has columns in this warp's group
        // moves to the next item with chunks (returns their number, 0 at the end)
        auto next_item = [&]() -> int {
            for (;;) {
                ci += gridDim.x;
                if (ci >= L.nitems) return 0;
                Item it;
                if (!item_at(L, ci, it)) continue;
                const int C = chunks_of(L, it);
                cols = it.n0 + cg * 32 < it.P->N;
                if (C > 0) return C;
            }
        };
        int left = next_item();
        int produced = 0, drained = 0;
        while (drained < total) {
            if (produced < total) {
                const int s = produced % NSTAGE, r = produced % NRAW;
                if (!mbar_wait(smem_u32(&rfull[r]), (uint32_t)((produced / NRAW) & 1), abort_flag) ||
                    (produced >= NSTAGE &&
                     !mbar_wait(smem_u32(&empty[s]), (uint32_t)((produced / NSTAGE - 1) & 1), abort_flag))) {
                    *abort_flag = 1;
                    break;
                }
                char* tile = smem + s * STAGE + (isB ? TILE : 0);
                const char* raw = smem + RAW_OFF + (2 * r + (isB ? 1 : 0)) * RAW_OP;
                const bool t = isB ? split_chunk<BMD == B_NK>(tile, raw, t8) : split_chunk<AM == A_MK>(tile, raw, t8);
                if (t) {
                    atomicMin(again, produced);
                    atomicMax(again + 1, produced);
                    *(volatile int*)(again + 4) = 1;
                }
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                __syncwarp();
                if (lane == 0) {
                    mbar_arrive(smem_u32(&full[s]));
                    mbar_arrive(smem_u32(&rempty[r]));
                }
                ++produced;
                if (produced < total && produced - drained <= LAG) continue;
            }
            const int b = drained & 1;
            if (!mbar_wait(smem_u32(&tfull[b]), (uint32_t)((drained >> 1) & 1), abort_flag)) {
                *abort_flag = 1;
                break;
            }
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            if (cols) {
#pragma unroll
                for (int h = 0; h < 4; ++h) {   // Re columns 0-15, 16-31, Im columns 0-15, 16-31
                    uint32_t r[16];
                    tmem_ld16(tm0 + b * 2 * TN + (h >> 1) * TN + (h & 1) * 16, r);
                    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
                    for (int j = 0; j < 8; ++j)
                        acc[h * 8 + j] =
                            add2(acc[h * 8 + j], pair(__uint_as_float(r[2 * j]), __uint_as_float(r[2 * j + 1])));
                }
            }
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&tempty[b]));
            ++drained;
            if (--left == 0) {
                Item it;
                item_at(L, ci, it);
                if (write_tile(L, it, acc, lg, cg, lane)) {
                    atomicMin(again + 2, ci);
                    atomicMax(again + 3, ci);
                    *(volatile int*)(again + 4) = 1;
                }
#pragma unroll
                for (int j = 0; j < 32; ++j) acc[j] = 0;
                left = next_item();
            }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (*abort_flag && threadIdx.x == 0) atomicExch(err, TLR_ERR_TIMEOUT);
    if (warp == WMMA) {
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(*tslot), "r"(TMEM_COLS) : "memory");
    }
    // what the split does not hold, and sums of few products
    if (warp < NW && again[4] && !*abort_flag) plain_items<AM, BMD>(L, again);
}

template <int AM, int BMD>
cudaError_t launch(const GemmLaunch& G, const Launch& L, unsigned grid, cudaStream_t st) {
    counted(1);
    if (t_early_blocks != kEarlyAny) {   // in a solve: a CTA takes a whole SM, early ones crowd (see chain_entry)
        k_cgemm_f32<AM, BMD><<<grid, NTHR, SMEM_BYTES, st>>>(L, G.err);
        return cudaGetLastError();
    }
    return launch_chain(k_cgemm_f32<AM, BMD>, dim3(grid), dim3(NTHR), SMEM_BYTES, st, L, G.err);
}

}  // namespace

int gemm_f32_split(long long tiles, long long K, long long most) {
    // the split s that minimises ceil(tiles s / SMs) (K / s + 48): whole waves of
    // tiles, each with a fixed cost (start of the pipeline, write-out) of about
    // 48 units of depth; at least 64 deep, so that a partial is worth its write
    const long long sms = device_sms(), smax = std::max(1LL, std::min({32LL, most, K / 64}));
    long long best = 1;
    double tbest = 1e300;
    for (long long s = 1; s <= smax; ++s) {
        const double t = (double)((std::max(1LL, tiles) * s + sms - 1) / sms) * ((double)K / s + 48.0);
        if (t < tbest * 0.98) {
            tbest = t;
            best = s;
        }
    }
    return (int)best;
}

cudaError_t gemm_f32_prepare() {
    cudaError_t e = cudaFuncSetAttribute(k_cgemm_f32<A_KM, B_KN>, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_BYTES);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_cgemm_f32<A_MK, B_KN>, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_BYTES);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_cgemm_f32<A_MK, B_NK>, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_BYTES);
    return e;
}

bool gemm_f32_shallow(const GProb& p, int nsplit, int kchunk) {
    for (int c = 0; c < nsplit; ++c) {
        long long d = 0;
        for (int t = 0; t < p.nt; ++t)
            d += nsplit == 1 ? p.t[t].K : std::max(0LL, std::min<long long>(p.t[t].K - (long long)c * kchunk, kchunk));
        if (d > 0 && d <= SHALLOW) return true;
    }
    return false;
}

cudaError_t gemm_f32(const GemmLaunch& G, cudaStream_t st) {
    if (G.nprob == 0 || G.maxM == 0 || G.maxN == 0) return cudaSuccess;
    if (!G.err || (G.epi != EPI_STORE && G.epi != EPI_SUB && G.epi != EPI_PARTIAL)) return cudaErrorInvalidValue;
    Launch L;
    L.probs = G.d_probs;
    L.nsplit = G.nsplit;
    L.kchunk = G.kchunk;
    L.nx = (G.maxN + TN - 1) / TN;
    L.ny = (G.maxM + TM - 1) / TM;
    const long long nitems = (long long)L.nx * L.ny * G.nprob * G.nsplit;
    if (nitems > 0x7fff0000LL) return cudaErrorInvalidValue;
    L.nitems = (int)nitems;
    L.epi = G.epi;
    L.shallow = G.shallow ? 1 : 0;
    L.part_stride = G.part_stride;
    const unsigned grid = (unsigned)std::min<long long>(device_sms(), nitems);
    if (G.amode == A_KM && G.bmode == B_KN) return launch<A_KM, B_KN>(G, L, grid, st);
    if (G.amode == A_MK && G.bmode == B_KN) return launch<A_MK, B_KN>(G, L, grid, st);
    if (G.amode == A_MK && G.bmode == B_NK) return launch<A_MK, B_NK>(G, L, grid, st);
    return cudaErrorInvalidValue;
}

}  // namespace tlr
