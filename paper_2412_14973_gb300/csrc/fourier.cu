// Time <-> frequency pipeline of the examples: the wavefields are recorded in
// time, transformed to the frequency domain and solved one frequency at a
// time; the Green's function comes back to time (time-offset gathers) by the
// inverse transform over the solved band.
//
// Traces are stored trace-major, x_t[tr][t] (tr = s nr + r for data, a nr +
// b for X), nt samples each.  X(omega_k) = sum_t x(t) exp(-2 pi i k t / nt)
// (unnormalised), k = 0 .. nt/2; the inverse puts the band [f0, f0 + nf) back
// (zero elsewhere) and divides by nt.
//
// Lengths up to 4096 with prime factors up to 13, and any length from 64 to 2048, take
// one kernel per direction: a CTA transforms a few pairs of traces (a pair as the
// real and imaginary part of one complex transform) in shared memory and writes
// the band of the frequency-major stack (stack[f][tr], one ns x nr panel per
// frequency) or the traces themselves, so a trace is read once and its band
// written once: 244 MB each way for 40000 traces of 1125 samples, 200 bins,
// where a library transform between a spectrum in memory and a gather moved
// 1.5 GB and its plans were made (and destroyed) on every call: 3.5 to 4.9 ms for both
// directions, as the host makes the plans, against 0.47 here (kernels 233 + 189 us).  Bound by shared-memory
// traffic (two passes per factor); the bytes alone would take 72 us.
//
// Other lengths: cuFFT plans over a chunk of traces, with the band gather /
// scatter between the trace-major spectrum and the stack as transposes through
// shared memory, coalesced on both sides.
#include <cufft.h>

#include <algorithm>
#include <cstring>
#include <string>

#include "internal.h"

namespace tlr {

namespace {

constexpr int FT = 32;

// out[f][tr] = spec[tr][f0 + f] for one chunk of traces (tr0 .. tr0 + ntr_c)
__global__ void __launch_bounds__(256) k_band_gather(const cf* __restrict__ spec, long long ntr_c, int nh, int f0,
                                                     int nf, cf* __restrict__ out, long long ld_out) {
    __shared__ cf t[FT][FT + 1];
    const long long tr0 = (long long)blockIdx.x * FT;
    const int fb = blockIdx.y * FT;
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    for (int r = ty; r < FT; r += 8) {
        const long long tr = tr0 + r;
        const int f = fb + tx;
        t[r][tx] = (tr < ntr_c && f < nf) ? spec[tr * nh + f0 + f] : make_float2(0.f, 0.f);
    }
    __syncthreads();
    for (int r = ty; r < FT; r += 8) {
        const int f = fb + r;
        const long long tr = tr0 + tx;
        if (f < nf && tr < ntr_c) out[(long long)f * ld_out + tr] = t[tx][r];
    }
}

// spec[tr][h] = in[h - f0][tr] inside the band, 0 outside, for one chunk
__global__ void __launch_bounds__(256) k_band_scatter(const cf* __restrict__ in, long long ld_in, long long ntr_c,
                                                      int nh, int f0, int nf, cf* __restrict__ spec) {
    __shared__ cf t[FT][FT + 1];
    const long long tr0 = (long long)blockIdx.x * FT;
    const int hb = blockIdx.y * FT;
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    for (int r = ty; r < FT; r += 8) {
        const int h = hb + r;
        const long long tr = tr0 + tx;
        const int f = h - f0;
        t[r][tx] = (tr < ntr_c && f >= 0 && f < nf) ? in[(long long)f * ld_in + tr] : make_float2(0.f, 0.f);
    }
    __syncthreads();
    for (int r = ty; r < FT; r += 8) {
        const long long tr = tr0 + r;
        const int h = hb + tx;
        if (tr < ntr_c && h < nh) spec[tr * nh + h] = t[tx][r];
    }
}

__global__ void k_scale(float* x, long long n, float s) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        x[i] *= s;
}

// ---------------------------------------------------------------------------
// transforms in shared memory
// ---------------------------------------------------------------------------
// A plan of length n: the complex transform has length M = n, factors fac[], or,
// for n with a prime factor above 13, M = a power of two >= 2 n - 1 (Bluestein
// 1970: the transform of n points as a convolution with a chirp).
constexpr int FFT_T = 256;
constexpr int FFT_MAXF = 12;
struct FftPlan {
    int n, M, nfac, B;             // B: trace pairs per CTA
    int exact;                     // the first factors, done exactly within the factor; the rest in plain FP32
    int lo;                        // offset of the tables' low parts
    int fac[FFT_MAXF];
    unsigned magic[FFT_MAXF];      // ceil(2^32 / L) of the stage's L = product of the factors before it
    unsigned magic_m[FFT_MAXF];    // ceil(2^32 / m), m = M / factor
    bool chirp;
};

// The tables of a plan: W_M^j = exp(-2 pi i j / M), j < M, then (chirp) c_t =
// exp(-pi i t^2 / n), t < n, then the transform of conj(c) wrapped to M (filled by
// k_fft_chirp), each FP64 value (the last: from two FP32 parts) rounded once; P.lo
// entries on, what the rounding left.
__global__ void k_fft_tables(FftPlan P, cf* __restrict__ tab) {
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    double s, c;
    if (e < P.M) {
        sincospi(-2.0 * e / P.M, &s, &c);
    } else if (P.chirp && e < P.M + P.n) {
        const long long t = e - P.M;
        sincospi(-(double)(t * t % (2LL * P.n)) / P.n, &s, &c);
    } else {
        return;
    }
    const cf h = make_float2((float)c, (float)s);
    tab[e] = h;
    tab[P.lo + e] = make_float2((float)(c - (double)h.x), (float)(s - (double)h.y));
}

__device__ __forceinline__ cf cmul(cf a, cf b) {
    return make_float2(fmaf(a.x, b.x, -a.y * b.y), fmaf(a.x, b.y, a.y * b.x));
}
__device__ __forceinline__ cf cadd(cf a, cf b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ cf csub(cf a, cf b) { return make_float2(a.x - b.x, a.y - b.y); }

// the transform of R values in place; W_R^1 = w[step] for the sizes without a
// closed form here
template <int R>
__device__ __forceinline__ void dft(cf* v, const cf* __restrict__ w, int step) {
    if (R == 2) {
        const cf a = v[0];
        v[0] = cadd(a, v[1]);
        v[1] = csub(a, v[1]);
    } else if (R == 4) {
        const cf a = cadd(v[0], v[2]), b = csub(v[0], v[2]), c = cadd(v[1], v[3]), d = csub(v[1], v[3]);
        v[0] = cadd(a, c);
        v[1] = make_float2(b.x + d.y, b.y - d.x);
        v[2] = csub(a, c);
        v[3] = make_float2(b.x - d.y, b.y + d.x);
    } else if (R == 3) {
        const cf s = cadd(v[1], v[2]), d = csub(v[1], v[2]);
        constexpr float h = 0.86602540378443864676f;   // sin(2 pi / 3)
        const cf m = make_float2(fmaf(-0.5f, s.x, v[0].x), fmaf(-0.5f, s.y, v[0].y));
        v[0] = cadd(v[0], s);
        v[1] = make_float2(fmaf(h, d.y, m.x), fmaf(-h, d.x, m.y));
        v[2] = make_float2(fmaf(-h, d.y, m.x), fmaf(h, d.x, m.y));
    } else if (R == 5) {
        constexpr float c1 = 0.30901699437494742410f, c2 = -0.80901699437494742410f;   // cos(2 pi / 5), cos(4 pi / 5)
        constexpr float s1 = 0.95105651629515357212f, s2 = 0.58778525229247312917f;    // sin(2 pi / 5), sin(4 pi / 5)
        const cf a = cadd(v[1], v[4]), b = csub(v[1], v[4]), c = cadd(v[2], v[3]), d = csub(v[2], v[3]);
        const cf p = make_float2(fmaf(c2, c.x, fmaf(c1, a.x, v[0].x)), fmaf(c2, c.y, fmaf(c1, a.y, v[0].y)));
        const cf q = make_float2(fmaf(c1, c.x, fmaf(c2, a.x, v[0].x)), fmaf(c1, c.y, fmaf(c2, a.y, v[0].y)));
        const cf r = make_float2(fmaf(s2, d.x, s1 * b.x), fmaf(s2, d.y, s1 * b.y));
        const cf t = make_float2(fmaf(-s1, d.x, s2 * b.x), fmaf(-s1, d.y, s2 * b.y));
        v[0] = cadd(v[0], cadd(a, c));
        v[1] = make_float2(p.x + r.y, p.y - r.x);
        v[4] = make_float2(p.x - r.y, p.y + r.x);
        v[2] = make_float2(q.x + t.y, q.y - t.x);
        v[3] = make_float2(q.x - t.y, q.y + t.x);
    } else {
        // pairs v_j +- v_{R-j}: real parts from the cosines, imaginary from the sines
        cf a[R / 2], b[R / 2], o[R];
        o[0] = v[0];
#pragma unroll
        for (int j = 0; j < R / 2; ++j) {
            a[j] = cadd(v[j + 1], v[R - 1 - j]);
            b[j] = csub(v[j + 1], v[R - 1 - j]);
            o[0] = cadd(o[0], a[j]);
        }
#pragma unroll
        for (int k = 1; k <= R / 2; ++k) {
            cf p = v[0], q = make_float2(0.f, 0.f);
#pragma unroll
            for (int j = 0; j < R / 2; ++j) {
                const cf t = w[(k * (j + 1) % R) * step];   // cos, -sin
                p = make_float2(fmaf(t.x, a[j].x, p.x), fmaf(t.x, a[j].y, p.y));
                q = make_float2(fmaf(-t.y, b[j].x, q.x), fmaf(-t.y, b[j].y, q.y));
            }
            o[k] = make_float2(p.x + q.y, p.y - q.x);
            o[R - k] = make_float2(p.x - q.y, p.y + q.x);
        }
#pragma unroll
        for (int k = 0; k < R; ++k) v[k] = o[k];
    }
}

// Exact within a factor: a complex value as the sum of two FP32 pairs (re, im), h
// the rounded value and l what it lacks, so that a factor's twiddle products, sums and
// constants leave one rounding, at its store.  In plain FP32 a factor rounds three to
// five times; where that gave more error than the library's transforms (see fft_plan)
// the factors are done like this: 14 packed instructions a twiddle, 8 a sum.
typedef unsigned long long f2;
__device__ __forceinline__ f2 pk(float x, float y) {
    f2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(x), "f"(y));
    return r;
}
__device__ __forceinline__ cf unpk(f2 a) {
    cf r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(a));
    return r;
}
__device__ __forceinline__ f2 add2(f2 a, f2 b) {
    f2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
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
__device__ __forceinline__ f2 sub2(f2 a, f2 b) { return fma2(b, pk(-1.f, -1.f), a); }   // one instruction
struct E2 {
    f2 h, l;
};
__device__ __forceinline__ E2 eadd(E2 a, E2 b) {   // Knuth's two-sum of the h, the l added
    const f2 s = add2(a.h, b.h), z = sub2(s, a.h);
    const f2 e = add2(sub2(a.h, sub2(s, z)), sub2(b.h, z));
    return E2{s, add2(e, add2(a.l, b.l))};
}
__device__ __forceinline__ E2 esub(E2 a, E2 b) {
    const f2 s = sub2(a.h, b.h), z = sub2(s, a.h);
    const f2 e = sub2(sub2(a.h, sub2(s, z)), add2(b.h, z));
    return E2{s, add2(e, sub2(a.l, b.l))};
}
// times the real c = ch + cl
__device__ __forceinline__ E2 escale(E2 a, float ch, float cl) {
    const f2 c = pk(ch, ch), p = mul2(a.h, c), n = mul2(a.h, pk(-ch, -ch));
    return E2{p, fma2(a.l, c, fma2(a.h, pk(cl, cl), fma2(a.h, c, n)))};
}
__device__ __forceinline__ f2 turn(f2 a) {   // times -i
    const cf v = unpk(a);
    return pk(v.y, -v.x);
}
__device__ __forceinline__ E2 eturn(E2 a) { return E2{turn(a.h), turn(a.l)}; }
__device__ __forceinline__ cf eround(E2 a) { return unpk(add2(a.h, a.l)); }
// v times the table value w + wl
__device__ __forceinline__ E2 emul(cf v, cf w, cf wl) {
    const f2 x = pk(v.x, v.x), y = pk(v.y, v.y), a = pk(w.x, w.y), b = pk(-w.y, w.x);
    const f2 p = mul2(x, a), q = mul2(y, b);
    const f2 e = add2(fma2(x, a, mul2(x, pk(-w.x, -w.y))), fma2(y, b, mul2(y, pk(w.y, -w.x))));
    const E2 r = eadd(E2{p, 0}, E2{q, 0});
    return E2{r.h, add2(add2(r.l, e), fma2(x, pk(wl.x, wl.y), mul2(y, pk(-wl.y, wl.x))))};
}
__device__ __forceinline__ float lo_of(double c) { return (float)(c - (double)(float)c); }

// the transform of R values (as dft); constants from the tables w, w + lo for 7, 11, 13
template <int R>
__device__ __forceinline__ void edft(E2* v, const cf* __restrict__ w, int lo, int step) {
    if (R == 2) {
        const E2 a = v[0];
        v[0] = eadd(a, v[1]);
        v[1] = esub(a, v[1]);
    } else if (R == 4) {
        const E2 a = eadd(v[0], v[2]), b = esub(v[0], v[2]), c = eadd(v[1], v[3]), d = eturn(esub(v[1], v[3]));
        v[0] = eadd(a, c);
        v[1] = eadd(b, d);
        v[2] = esub(a, c);
        v[3] = esub(b, d);
    } else if (R == 3) {
        constexpr double h = 0.86602540378443864676;   // sin(2 pi / 3)
        const E2 s = eadd(v[1], v[2]), d = eturn(escale(esub(v[1], v[2]), (float)h, lo_of(h)));
        const E2 m = eadd(v[0], escale(s, -0.5f, 0.f));
        v[0] = eadd(v[0], s);
        v[1] = eadd(m, d);
        v[2] = esub(m, d);
    } else if (R == 5) {
        constexpr double c1 = 0.30901699437494742410, c2 = -0.80901699437494742410;
        constexpr double s1 = 0.95105651629515357212, s2 = 0.58778525229247312917;
        const E2 a = eadd(v[1], v[4]), b = esub(v[1], v[4]), c = eadd(v[2], v[3]), d = esub(v[2], v[3]);
        const E2 p = eadd(v[0], eadd(escale(a, (float)c1, lo_of(c1)), escale(c, (float)c2, lo_of(c2))));
        const E2 q = eadd(v[0], eadd(escale(a, (float)c2, lo_of(c2)), escale(c, (float)c1, lo_of(c1))));
        const E2 r = eturn(eadd(escale(b, (float)s1, lo_of(s1)), escale(d, (float)s2, lo_of(s2))));
        const E2 t = eturn(esub(escale(b, (float)s2, lo_of(s2)), escale(d, (float)s1, lo_of(s1))));
        v[0] = eadd(v[0], eadd(a, c));
        v[1] = eadd(p, r);
        v[4] = esub(p, r);
        v[2] = eadd(q, t);
        v[3] = esub(q, t);
    } else {
        E2 a[R / 2], b[R / 2], o[R];
        o[0] = v[0];
#pragma unroll
        for (int j = 0; j < R / 2; ++j) {
            a[j] = eadd(v[j + 1], v[R - 1 - j]);
            b[j] = eturn(esub(v[j + 1], v[R - 1 - j]));
            o[0] = eadd(o[0], a[j]);
        }
#pragma unroll
        for (int k = 1; k <= R / 2; ++k) {
            E2 p = v[0], q = E2{0, 0};
#pragma unroll
            for (int j = 0; j < R / 2; ++j) {
                const int i = (k * (j + 1) % R) * step;
                const cf t = __ldg(w + i), u = __ldg(w + lo + i);   // cos, -sin
                p = eadd(p, escale(a[j], t.x, u.x));
                q = eadd(q, escale(b[j], -t.y, -u.y));
            }
            o[k] = eadd(p, q);
            o[R - k] = esub(p, q);
        }
#pragma unroll
        for (int k = 0; k < R; ++k) v[k] = o[k];
    }
}

// one factor of `count` transforms of length M (rows of ld values): Stockham's
// autosort step, src to dst.  The butterflies of all rows share the threads.
// up != nullptr: the two parts of row b's values times up[2 b], up[2 b + 1] first.
template <int R, bool EX>
__device__ __forceinline__ void fft_stage(const cf* __restrict__ src, cf* __restrict__ dst, int M, int ld, int count,
                                          int L, unsigned magic, unsigned magic_m, const cf* __restrict__ w, int lo,
                                          const float* up) {
    const int m = M / R, step = m / L;   // step: W_{L R}^1 = W_M^step
    for (int e = threadIdx.x; e < count * m; e += FFT_T) {
        const int b = m == 1 ? e : (int)__umulhi((unsigned)e, magic_m), j = e - b * m;
        const int g = L == 1 ? j : (int)__umulhi((unsigned)j, magic), k = j - g * L;
        const cf* s = src + b * ld + j;
        cf v[R];
#pragma unroll
        for (int q = 0; q < R; ++q) v[q] = s[q * m];
        if (up) {
            const float ux = up[2 * b], uy = up[2 * b + 1];
#pragma unroll
            for (int q = 0; q < R; ++q) v[q] = make_float2(v[q].x * ux, v[q].y * uy);
        }
        if (EX) {
            E2 x[R];
            x[0] = E2{pk(v[0].x, v[0].y), 0};
#pragma unroll
            for (int q = 1; q < R; ++q) {
                if (k)
                    x[q] = emul(v[q], __ldg(w + k * q * step), __ldg(w + lo + k * q * step));
                else
                    x[q] = E2{pk(v[q].x, v[q].y), 0};
            }
            edft<R>(x, w, lo, m);
#pragma unroll
            for (int q = 0; q < R; ++q) v[q] = eround(x[q]);
        } else {
            if (k) {
#pragma unroll
                for (int q = 1; q < R; ++q) v[q] = cmul(v[q], __ldg(w + k * q * step));
            }
            dft<R>(v, w, m);
        }
        cf* d = dst + b * ld + g * L * R + k;
#pragma unroll
        for (int q = 0; q < R; ++q) d[q * L] = v[q];
    }
    __syncthreads();
}

template <bool EX>
__device__ __forceinline__ void fft_factor(const FftPlan& P, int f, const cf* a, cf* b, int ld, int count, int L,
                                           const cf* __restrict__ w, const float* up) {
    const unsigned mg = P.magic[f], mm = P.magic_m[f];
    switch (P.fac[f]) {
        case 2: fft_stage<2, EX>(a, b, P.M, ld, count, L, mg, mm, w, P.lo, up); break;
        case 3: fft_stage<3, EX>(a, b, P.M, ld, count, L, mg, mm, w, P.lo, up); break;
        case 4: fft_stage<4, EX>(a, b, P.M, ld, count, L, mg, mm, w, P.lo, up); break;
        case 5: fft_stage<5, EX>(a, b, P.M, ld, count, L, mg, mm, w, P.lo, up); break;
        case 7: fft_stage<7, EX>(a, b, P.M, ld, count, L, mg, mm, w, P.lo, up); break;
        case 11: fft_stage<11, EX>(a, b, P.M, ld, count, L, mg, mm, w, P.lo, up); break;
        default: fft_stage<13, EX>(a, b, P.M, ld, count, L, mg, mm, w, P.lo, up); break;
    }
}

// `count` transforms of length M in a (scratch b), their parts times up[] first
// (up != nullptr); returns where they end up
template <bool EX>
__device__ __forceinline__ cf* fft_rows(const FftPlan& P, cf* a, cf* b, int ld, int count, const cf* __restrict__ w,
                                        const float* up) {
    int L = 1;
    for (int f = 0; f < P.nfac; ++f) {
        if (EX && f < P.exact)
            fft_factor<true>(P, f, a, b, ld, count, L, w, up);
        else
            fft_factor<false>(P, f, a, b, ld, count, L, w, up);
        up = nullptr;
        L *= P.fac[f];
        cf* t = a;
        a = b;
        b = t;
    }
    return a;
}

// v times the table entry i
template <bool EX>
__device__ __forceinline__ cf tmul(cf v, const cf* __restrict__ tab, int lo, int i) {
    return EX ? eround(emul(v, __ldg(tab + i), __ldg(tab + lo + i))) : cmul(v, __ldg(tab + i));
}

// the n-point transforms of the rows of a (n values each, zeros beyond them when
// P.chirp): plain, or by the chirp convolution
template <bool EX>
__device__ __forceinline__ cf* fft_any(const FftPlan& P, cf* a, cf* b, int ld, const cf* __restrict__ tab,
                                       const float* up) {
    if (!P.chirp && (P.nfac || !up)) return fft_rows<EX>(P, a, b, ld, P.B, tab, up);
    if (!P.chirp) {   // one point
        const int r = threadIdx.x;
        if (r < P.B) a[r * ld] = make_float2(a[r * ld].x * up[2 * r], a[r * ld].y * up[2 * r + 1]);
        __syncthreads();
        return a;
    }
    const cf* c = tab + P.M;
    const cf* bt = c + P.n;
    cf* y = fft_rows<EX>(P, a, b, ld, P.B, tab, nullptr);
    for (int r = 0; r < P.B; ++r)
        for (int k = threadIdx.x; k < P.M; k += FFT_T) {
            const cf t = tmul<EX>(y[r * ld + k], bt, P.lo, k);
            y[r * ld + k] = make_float2(t.x, -t.y);   // conjugated: the inverse by a forward transform
        }
    __syncthreads();
    y = fft_rows<EX>(P, y, y == a ? b : a, ld, P.B, tab, nullptr);
    const float s = 1.f / (float)P.M;
    for (int r = 0; r < P.B; ++r)
        for (int k = threadIdx.x; k < P.n; k += FFT_T) {
            const cf t = y[r * ld + k];
            y[r * ld + k] = tmul<EX>(make_float2(t.x * s, -t.y * s), c, P.lo, k);
        }
    __syncthreads();
    return y;
}

// The transform of the wrapped conjugate chirp, for P.chirp (one CTA; factors 4 and
// 2), with both parts of every value kept: it multiplies every trace, so its
// roundings would be an error that all of them share.
template <int R>
__device__ __forceinline__ void chirp_stage(const cf* sh, const cf* sl, cf* dh, cf* dl, int M, int L, int lo,
                                            const cf* __restrict__ w) {
    const int m = M / R, step = m / L;
    for (int j = threadIdx.x; j < m; j += FFT_T) {
        const int g = j / L, k = j - g * L;
        E2 x[R];
#pragma unroll
        for (int q = 0; q < R; ++q) {
            const cf h = sh[q * m + j], l = sl[q * m + j], t = __ldg(w + k * q * step);
            x[q] = emul(h, t, __ldg(w + lo + k * q * step));
            x[q].l = add2(x[q].l, fma2(pk(l.x, l.x), pk(t.x, t.y), mul2(pk(l.y, l.y), pk(-t.y, t.x))));
        }
        edft<R>(x, w, lo, m);
#pragma unroll
        for (int q = 0; q < R; ++q) {
            const f2 h = add2(x[q].h, x[q].l);
            dh[g * L * R + k + q * L] = unpk(h);
            dl[g * L * R + k + q * L] = unpk(sub2(x[q].l, sub2(h, x[q].h)));
        }
    }
    __syncthreads();
}

__global__ void __launch_bounds__(FFT_T) k_fft_chirp(const __grid_constant__ FftPlan P, cf* __restrict__ tab) {
    extern __shared__ __align__(16) cf sm[];
    const int M = P.M;
    const cf* c = tab + M;
    cf *h = sm, *l = h + M, *h2 = l + M, *l2 = h2 + M;
    for (int k = threadIdx.x; k < M; k += FFT_T) {
        const int t = min(k, M - k);
        cf v = make_float2(0.f, 0.f), u = v;
        if (t < P.n) {
            v = make_float2(c[t].x, -c[t].y);
            u = make_float2(c[P.lo + t].x, -c[P.lo + t].y);
        }
        h[k] = v;
        l[k] = u;
    }
    __syncthreads();
    int L = 1;
    for (int f = 0; f < P.nfac; ++f) {
        if (P.fac[f] == 4)
            chirp_stage<4>(h, l, h2, l2, M, L, P.lo, tab);
        else
            chirp_stage<2>(h, l, h2, l2, M, L, P.lo, tab);
        L *= P.fac[f];
        cf* t = h;
        h = h2, h2 = t;
        t = l;
        l = l2, l2 = t;
    }
    for (int k = threadIdx.x; k < M; k += FFT_T) {
        tab[M + P.n + k] = h[k];
        tab[P.lo + M + P.n + k] = l[k];
    }
}

// The two traces of a pair share a transform, so each is scaled by a power of
// two to about unit 2-norm first (exact, undone on the results: the error of
// either stays relative to its own norm, and a trace of zeros stays zeros).
// From every thread's squared norms s1, s2 over values of its pair (n1, n2: any
// of them not zero): the scales up[], down[] per trace of the CTA.  Lanes `b` apart
// share a pair (warp: one pair per warp).  Returns whether a trace's norm is not to
// be had (Inf, NaN, or a squared norm outside 1e-30 .. 1e30): then the traces are
// transformed one at a time, such a one scaled by 2^-64 or 2^64, which keeps the
// chirp's sums in range.
__device__ __forceinline__ bool pair_scales(float s1, float s2, bool n1, bool n2, int pair, int apart_by, int B,
                                            float* up, float* down) {
    __shared__ float red[FFT_T / 32][16], nzr[FFT_T / 32][16];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (lane < 16) red[w][lane] = nzr[w][lane] = 0.f;
    __syncwarp();
    float z1 = n1 ? 1.f : 0.f, z2 = n2 ? 1.f : 0.f;
    for (int o = 16; o >= apart_by; o >>= 1) {
        s1 += __shfl_xor_sync(0xffffffffu, s1, o);
        s2 += __shfl_xor_sync(0xffffffffu, s2, o);
        z1 += __shfl_xor_sync(0xffffffffu, z1, o);
        z2 += __shfl_xor_sync(0xffffffffu, z2, o);
    }
    if (lane < apart_by) {
        red[w][2 * pair] = s1;
        red[w][2 * pair + 1] = s2;
        nzr[w][2 * pair] = z1;
        nzr[w][2 * pair + 1] = z2;
    }
    __syncthreads();
    bool odd = false;
    if (threadIdx.x < 2 * B) {
        float ss = 0.f, nz = 0.f;
        for (int i = 0; i < FFT_T / 32; ++i) {
            ss += red[i][threadIdx.x];
            nz += nzr[i][threadIdx.x];
        }
        odd = nz != 0.f && !(ss > 1e-30f && ss < 1e30f);
        const int e = nz == 0.f ? 0 : !odd ? ilogbf(ss) / 2 : ss <= 1e-30f ? -64 : 64;
        up[threadIdx.x] = ldexpf(1.f, -e);
        down[threadIdx.x] = nz != 0.f ? ldexpf(1.f, e) : 0.f;
    }
    return __syncthreads_or(odd) != 0;
}

// stack[f][tr] = the bins f0 .. f0 + nf - 1 of the traces; a CTA takes P.B pairs
template <bool EX>
__global__ void __launch_bounds__(FFT_T, 3)
    k_fft_forward(const __grid_constant__ FftPlan P, const float* __restrict__ x, long long ntr, int f0, int nf,
                  const cf* __restrict__ tab, cf* __restrict__ out) {
    extern __shared__ __align__(16) cf sm[];
    __shared__ float up[16], down[16];
    const int n = P.n, ld = P.M + 1, B = P.B;   // odd row length: a bin's rows lie in different banks
    const long long t0 = (long long)blockIdx.x * 2 * B;
    cf* a = sm;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // a warp loads one pair (8 / B warps share it).  pass -1: both traces; 0, 1:
    // the first, the second alone
    const int pr = warp & (B - 1);
    float s1 = 0.f, s2 = 0.f;
    bool n1 = false, n2 = false;
    auto load = [&](int pass) {
        const long long tr = t0 + 2 * pr;
        const bool in1 = tr < ntr && pass != 1, in2 = tr + 1 < ntr && pass != 0;
        const float* xa = x + tr * n;
        const float* xb = xa + n;
#pragma unroll 4
        for (int t = warp / B * 32 + lane; t < P.M; t += FFT_T / B) {
            cf v = make_float2(in1 && t < n ? xa[t] : 0.f, in2 && t < n ? xb[t] : 0.f);
            s1 = fmaf(v.x, v.x, s1);
            s2 = fmaf(v.y, v.y, s2);
            n1 = n1 || v.x != 0.f;
            n2 = n2 || v.y != 0.f;
            if (pass == 0) v.x *= up[2 * pr];
            if (pass == 1) v = make_float2(v.y * up[2 * pr + 1], 0.f);
            a[pr * ld + t] = v;
        }
    };
    load(-1);
    const bool apart = pair_scales(s1, s2, n1, n2, pr, 1, B, up, down);
    const bool vec = (ntr & 1) == 0 && (reinterpret_cast<uintptr_t>(out) & 15) == 0;
    for (int pass = apart ? 0 : -1; pass < (apart ? 2 : 0); ++pass) {
        if (apart) {
            load(pass);
            __syncthreads();
        }
        if (P.chirp) {
            for (int b = 0; b < B; ++b)
                for (int t = threadIdx.x; t < n; t += FFT_T) {
                    cf v = a[b * ld + t];
                    if (!apart) v = make_float2(v.x * up[2 * b], v.y * up[2 * b + 1]);
                    a[b * ld + t] = tmul<EX>(v, tab + P.M, P.lo, t);
                }
            __syncthreads();
        }
        const cf* z = fft_any<EX>(P, a, sm + B * ld, ld, tab, apart ? nullptr : up);
        for (int e = threadIdx.x; e < nf * B; e += FFT_T) {
            const int b = e & (B - 1), f = e / B;   // B is 8, 4 or 2
            const int k = f0 + f, kc = k == 0 ? 0 : n - k;
            const cf u = z[b * ld + k], v = z[b * ld + kc];
            const long long tr = t0 + 2 * b, o = (long long)f * ntr + tr;
            if (apart) {
                const float h = down[2 * b + pass];
                if (tr + pass < ntr) out[o + pass] = make_float2(u.x * h, u.y * h);
                continue;
            }
            // z = x1 + i x2: X1 = (Z_k + conj Z_{n-k}) / 2, X2 = (Z_k - conj Z_{n-k}) / 2i
            const float h1 = 0.5f * down[2 * b], h2 = 0.5f * down[2 * b + 1];
            const cf p = make_float2(h1 * (u.x + v.x), h1 * (u.y - v.y));
            const cf q = make_float2(h2 * (u.y + v.y), h2 * (v.x - u.x));
            if (vec && tr < ntr) {
                *reinterpret_cast<float4*>(out + o) = make_float4(p.x, p.y, q.x, q.y);
            } else {
                if (tr < ntr) out[o] = p;
                if (tr + 1 < ntr) out[o + 1] = q;
            }
        }
        __syncthreads();
    }
}

// traces from the bins f0 .. f0 + nf - 1 (zero elsewhere, the imaginary parts of
// bins 0 and n / 2 ignored), times 1 / n.  The band is read twice, once for the
// norms (the second time from L2).
template <bool EX>
__global__ void __launch_bounds__(FFT_T, 3)
    k_fft_inverse(const __grid_constant__ FftPlan P, const cf* __restrict__ in, long long ntr, int f0, int nf,
                  const cf* __restrict__ tab, float* __restrict__ x) {
    extern __shared__ __align__(16) cf sm[];
    __shared__ float up[16], down[16];
    const int n = P.n, ld = P.M + 1, B = P.B;
    const long long t0 = (long long)blockIdx.x * 2 * B;
    const int b = threadIdx.x & (B - 1), fs = FFT_T / B;   // a thread's pair and its step over bins
    const long long tr = t0 + 2 * b;
    const bool vec = (ntr & 1) == 0 && (reinterpret_cast<uintptr_t>(in) & 15) == 0;
    auto bin = [&](int f, cf& p, cf& q) {
        const long long o = (long long)f * ntr + tr;
        p = q = make_float2(0.f, 0.f);
        if (vec && tr < ntr) {
            const float4 v = *reinterpret_cast<const float4*>(in + o);
            p = make_float2(v.x, v.y);
            q = make_float2(v.z, v.w);
        } else {
            if (tr < ntr) p = in[o];
            if (tr + 1 < ntr) q = in[o + 1];
        }
        const int k = f0 + f;
        if (k == 0 || 2 * k == n) p.y = q.y = 0.f;
    };
    bool apart;
    {
        float s1 = 0.f, s2 = 0.f;
        bool n1 = false, n2 = false;
#pragma unroll 4
        for (int f = threadIdx.x / B; f < nf; f += fs) {
            cf p, q;
            bin(f, p, q);
            s1 = fmaf(p.x, p.x, fmaf(p.y, p.y, s1));
            s2 = fmaf(q.x, q.x, fmaf(q.y, q.y, s2));
            n1 = n1 || p.x != 0.f || p.y != 0.f;
            n2 = n2 || q.x != 0.f || q.y != 0.f;
        }
        apart = pair_scales(s1, s2, n1, n2, b, B, B, up, down);
    }
    // v / n: a product with the rounded 1 / n would be an error that all values share
    const float s = 1.f / (float)n, nn = (float)n;
    auto over_n = [&](float v) {
        const float q = v * s;
        return fmaf(fmaf(-q, nn, v), s, q);
    };
    for (int pass = apart ? 0 : -1; pass < (apart ? 2 : 0); ++pass) {
        for (int e = threadIdx.x; e < B * ld; e += FFT_T) sm[e] = make_float2(0.f, 0.f);
        __syncthreads();
        for (int f = threadIdx.x / B; f < nf; f += fs) {
            cf p, q;
            bin(f, p, q);
            if (apart) {
                if (pass == 1) p = q;
                p = make_float2(p.x * up[2 * b + pass], p.y * up[2 * b + pass]);
                q = make_float2(0.f, 0.f);
            } else {   // the spectra are scaled here: a bin mixes both traces
                p = make_float2(p.x * up[2 * b], p.y * up[2 * b]);
                q = make_float2(q.x * up[2 * b + 1], q.y * up[2 * b + 1]);
            }
            const int k = f0 + f;
            // conj(Z_k) with Z = X1 + i X2, and conj(Z_{n-k}) from X_{n-k} = conj X_k
            cf u = make_float2(p.x - q.y, -(p.y + q.x)), w = make_float2(p.x + q.y, p.y - q.x);
            if (P.chirp) u = tmul<EX>(u, tab + P.M, P.lo, k);
            sm[b * ld + k] = u;
            if (k > 0 && 2 * k < n) {
                if (P.chirp) w = tmul<EX>(w, tab + P.M, P.lo, n - k);
                sm[b * ld + n - k] = w;
            }
        }
        __syncthreads();
        const cf* z = fft_any<EX>(P, sm, sm + B * ld, ld, tab, nullptr);
        for (int r = 0; r < B; ++r) {
            float* xa = x + (t0 + 2 * r) * n;
            float* xb = xa + n;
            const bool in1 = t0 + 2 * r < ntr, in2 = t0 + 2 * r + 1 < ntr;
            for (int t = threadIdx.x; t < n; t += FFT_T) {
                const cf v = z[r * ld + t];   // the conjugate of n (x1 + i x2)
                if (apart) {
                    if (pass ? in2 : in1) (pass ? xb : xa)[t] = over_n(v.x) * down[2 * r + pass];
                } else {
                    if (in1) xa[t] = over_n(v.x) * down[2 * r];
                    if (in2) xb[t] = over_n(-v.y) * down[2 * r + 1];
                }
            }
        }
        __syncthreads();
    }
}

// How many of a transform's factors are done exactly: where plain FP32 gives a larger
// error than the library's transforms, as many as bring it below.  Measured against 64
// bits, white traces, own / library, over every length with factors to 13 up to 4096
// and 560 others up to 2048.  Plain: powers of two from 64 on 0.66 to 0.9; forward
// 0.5 to 0.95 from length 100 on (up to 1.2 below); inverse 0.5 to 1.0 for even lengths
// above 1296 and odd ones from 1000 on but powers of a prime (1.09 at 3125), up to 1.22
// below (1.036 at 1080); chirps 0.6 to 0.77 where the largest prime factor is above 127,
// up to 1.64 where the library has factors for it (1.18 from 1024 on).  So: 0.45 to 1.0.
// Both ways over 45 million samples: 720 points 0.66 -> 0.92 ms (the library 1.38), the
// chirp of 247 points 1.74 -> 3.45 (4.07); over 0.4 million 0.060 -> 0.067 and 0.093 ->
// 0.125 (its plans, made on every call, take 1.8 ms of the host).
int exact_factors(const FftPlan& P, bool forward) {
    int most = 0, rest = P.n;
    for (int f = 2; f * f <= rest; ++f)
        while (rest % f == 0) {
            most = f;
            rest /= f;
        }
    if (rest > 1) most = std::max(most, rest);   // the largest prime factor
    if (P.chirp) {
        if (most > 127) return 0;
        return P.n < 1024 ? P.nfac : (P.nfac + 1) / 2;
    }
    if (P.n < 64) return P.nfac;
    if (most == 2) return 0;
    if (forward) return P.n < 100 ? P.nfac : 0;
    bool power = true;   // of one odd prime
    for (int f = 1; f < P.nfac; ++f) power = power && P.fac[f] == P.fac[0];
    const bool low = P.n % 2 == 0 ? P.n <= 1296 : P.n < 1000;
    return low || (power && P.n % 2) ? (2 * P.nfac + 2) / 3 : 0;
}

// The plan of length n; false: not a length for these kernels.
bool fft_plan(long long n, bool forward, FftPlan& P) {
    if (n < 1 || n > 4096) return false;
    memset(&P, 0, sizeof(P));
    P.n = (int)n;
    auto factor = [&](int m) {
        P.nfac = 0;
        unsigned long long L = 1;
        for (int f : {13, 11, 7, 5, 3, 4, 2})   // odd factors first: their strides meet no bank conflicts
            while (m % f == 0) {
                P.fac[P.nfac] = f;
                P.magic[P.nfac++] = L == 1 ? 0u : (unsigned)(((1ull << 32) + L - 1) / L);
                m /= f;
                L *= f;
            }
        for (int f = 0; m == 1 && f < P.nfac; ++f) {
            const unsigned long long k = L / P.fac[f];
            P.magic_m[f] = k == 1 ? 0u : (unsigned)(((1ull << 32) + k - 1) / k);
        }
        return m == 1;
    };
    P.M = P.n;
    if (!factor(P.n)) {
        if (n > 2048) return false;
        P.chirp = true;
        P.M = 1;
        while (P.M < 2 * P.n - 1) P.M *= 2;
        factor(P.M);
    }
    P.lo = P.M + (P.chirp ? P.n + P.M : 0);
    P.exact = exact_factors(P, forward);
    // trace pairs per CTA: the most of 8, 4 that leave room for three CTAs per SM, else 2
    P.B = 8;
    while (P.B > 2 && 2 * P.B * (P.M + 1) * (int)sizeof(cf) > 74 * 1024) P.B /= 2;
    return true;
}

// both directions in shared memory (see the top of this file)
int fft_shared(const FftPlan& P, bool forward, const float* x_in, const cf* X_in, long long ntr, long long f0,
               long long nf, cf* X_out, float* x_out, char* scratch, cudaStream_t st, std::string& err) {
    cf* tab = reinterpret_cast<cf*>(scratch);
    const int smem = 2 * P.B * (P.M + 1) * (int)sizeof(cf);
    const int entries = P.M + (P.chirp ? P.n : 0);
    const long long ctas = (ntr + 2 * P.B - 1) / (2 * P.B);
    constexpr int most = 2 * 2 * 4097 * (int)sizeof(cf);
    const bool ex = P.exact > 0;
    const void* kernel = forward ? (ex ? (const void*)k_fft_forward<true> : (const void*)k_fft_forward<false>)
                                 : (ex ? (const void*)k_fft_inverse<true> : (const void*)k_fft_inverse<false>);
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_fft_chirp, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
    if (e == cudaSuccess) {
        k_fft_tables<<<(entries + 63) / 64, 64, 0, st>>>(P, tab);
        if (P.chirp) k_fft_chirp<<<1, FFT_T, 4 * P.M * (int)sizeof(cf), st>>>(P, tab);
        if (forward && ex)
            k_fft_forward<true><<<(unsigned)ctas, FFT_T, smem, st>>>(P, x_in, ntr, (int)f0, (int)nf, tab, X_out);
        else if (forward)
            k_fft_forward<false><<<(unsigned)ctas, FFT_T, smem, st>>>(P, x_in, ntr, (int)f0, (int)nf, tab, X_out);
        else if (ex)
            k_fft_inverse<true><<<(unsigned)ctas, FFT_T, smem, st>>>(P, X_in, ntr, (int)f0, (int)nf, tab, x_out);
        else
            k_fft_inverse<false><<<(unsigned)ctas, FFT_T, smem, st>>>(P, X_in, ntr, (int)f0, (int)nf, tab, x_out);
        counted(P.chirp ? 3 : 2);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) {
        err = cudaGetErrorString(e);
        return TLR_ERR_CUDA;
    }
    return TLR_OK;
}

const char* cufft_msg(cufftResult r) {
    switch (r) {
        case CUFFT_SUCCESS: return "success";
        case CUFFT_ALLOC_FAILED: return "cuFFT allocation failed";
        case CUFFT_INVALID_VALUE: return "cuFFT invalid value";
        case CUFFT_EXEC_FAILED: return "cuFFT execution failed";
        case CUFFT_SETUP_FAILED: return "cuFFT setup failed";
        case CUFFT_INVALID_SIZE: return "cuFFT invalid size";
        default: return "cuFFT error";
    }
}

// traces per chunk: the chunk's real and complex buffers within ~256 MB; an even
// number of them, so that every chunk starts on 8 bytes like the first (cuFFT refuses
// real arrays that do not)
long long chunk_traces(long long ntr, long long nt) {
    const long long per = nt * 4 + (nt / 2 + 1) * 8;
    long long c = std::max(1LL, (256LL << 20) / per);
    return std::min(ntr, c + (c & 1));
}

}  // namespace

size_t fft_scratch_bytes(long long nt) {
    FftPlan P;
    return fft_plan(nt, true, P) ? 2 * (size_t)P.lo * sizeof(cf) : 0;
}

static int fft_library(bool forward, const float* x_t_in, const cf* X_in, long long ntr, long long nt, long long f0,
                       long long nf, cf* X_out, float* x_t_out, cudaStream_t st, std::string& err) {
    const long long nh = nt / 2 + 1;
    const long long C = chunk_traces(ntr, nt);
    cf* spec = nullptr;
    cudaError_t e = cudaMallocAsync((void**)&spec, (size_t)C * nh * sizeof(cf), st);
    if (e != cudaSuccess) {
        err = std::string("frequency stack: ") + cudaGetErrorString(e);
        return e == cudaErrorMemoryAllocation ? TLR_ERR_NOMEM : TLR_ERR_CUDA;
    }
    int rc = TLR_OK;
    cufftHandle plan = 0, plan_tail = 0;
    long long planned = 0, planned_tail = 0;
    for (long long tr0 = 0; tr0 < ntr && rc == TLR_OK; tr0 += C) {
        const long long c = std::min(C, ntr - tr0);
        cufftHandle* p = c == C ? &plan : &plan_tail;
        long long& have = c == C ? planned : planned_tail;
        if (have != c) {
            int n[1] = {(int)nt};
            const cufftResult r = cufftPlanMany(p, 1, n, nullptr, 1, (int)nt, nullptr, 1, (int)nh,
                                                forward ? CUFFT_R2C : CUFFT_C2R, (int)c);
            if (r != CUFFT_SUCCESS) {
                err = cufft_msg(r);
                rc = r == CUFFT_ALLOC_FAILED ? TLR_ERR_NOMEM : TLR_ERR_CUDA;
                break;
            }
            cufftSetStream(*p, st);
            have = c;
        }
        const dim3 grid((unsigned)((c + FT - 1) / FT), (unsigned)(((forward ? nf : nh) + FT - 1) / FT));
        cufftResult r;
        if (forward) {
            r = cufftExecR2C(*p, const_cast<float*>(x_t_in) + tr0 * nt, reinterpret_cast<cufftComplex*>(spec));
            if (r == CUFFT_SUCCESS) {
                k_band_gather<<<grid, 256, 0, st>>>(spec, c, (int)nh, (int)f0, (int)nf, X_out + tr0, ntr);
                counted(1);
            }
        } else {
            k_band_scatter<<<grid, 256, 0, st>>>(X_in + tr0, ntr, c, (int)nh, (int)f0, (int)nf, spec);
            counted(1);
            r = cufftExecC2R(*p, reinterpret_cast<cufftComplex*>(spec), x_t_out + tr0 * nt);
            if (r == CUFFT_SUCCESS) {
                k_scale<<<1024, 256, 0, st>>>(x_t_out + tr0 * nt, c * nt, 1.f / (float)nt);
                counted(1);
            }
        }
        if (r != CUFFT_SUCCESS) {
            err = cufft_msg(r);
            rc = TLR_ERR_CUDA;
        } else if ((e = cudaGetLastError()) != cudaSuccess) {
            err = cudaGetErrorString(e);
            rc = TLR_ERR_CUDA;
        }
    }
    if (e == cudaSuccess && rc == TLR_OK) e = cudaStreamSynchronize(st);   // plans are destroyed below
    if (e != cudaSuccess && rc == TLR_OK) {
        err = cudaGetErrorString(e);
        rc = TLR_ERR_CUDA;
    }
    if (plan) cufftDestroy(plan);
    if (plan_tail) cufftDestroy(plan_tail);
    cudaFreeAsync(spec, st);
    return rc;
}

int fft_stack(bool forward, const float* x_t_in, const cf* X_in, long long ntr, long long nt, long long f0,
              long long nf, cf* X_out, float* x_t_out, char* scratch, cudaStream_t st, std::string& err) {
    FftPlan P;
    const bool own = scratch && fft_plan(nt, forward, P) && ntr <= 0x7fffffffLL;
    // short chirps are left to the library, whose factors reach to 127 (17, 19 and 23 points:
    // own error up to 1.06 times its); it takes real arrays that start on 8 bytes
    const bool aligned = (reinterpret_cast<uintptr_t>(forward ? x_t_in : x_t_out) & 7) == 0;
    if (!own || (aligned && P.chirp && P.n < 64)) {
        const int rc = fft_library(forward, x_t_in, X_in, ntr, nt, f0, nf, X_out, x_t_out, st, err);
        if (!own || rc != TLR_ERR_NOMEM) return rc;
        (void)cudaGetLastError();   // no room for its work memory
        err.clear();
    }
    return fft_shared(P, forward, x_t_in, X_in, ntr, f0, nf, X_out, x_t_out, scratch, st, err);
}

}  // namespace tlr
