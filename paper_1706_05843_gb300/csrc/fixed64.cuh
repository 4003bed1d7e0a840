// fixed64.cuh -- the FP64 Wilson hop in 64-bit fixed point on the integer pipe.
//
// GB300 issues 1.9 FP64 lanes per clock and SM (measured; one warp
// instruction every 17 clocks) but 60 lanes of 32 x 32 + 64 bit integer
// multiply-adds (mad.wide.s32), so the SU(3) products of the FP64 hop are
// integer work here:
//
//  * a spinor that a hop reads is kept in memory as 24 signed integers in
//    units of 2^(E-56) and E, the exponent field of its largest real (fx_pack,
//    by the kernel that makes it): 57 bits, so every real within 2^-4 of the
//    largest is exact and the others are rounded to half a unit, 2^-5 of the
//    ulp of the largest;
//  * spin projection and reconstruction are 64-bit integer additions (exact);
//  * a link's reals are 58-bit fixed point (Uh, Ul): u = (Uh 2^29 + Ul) 2^-58,
//    |Ul| <= 2^28; a projected component is H = Hh 2^29 + Hl likewise, and
//    U H = sum Uh Hh + 2^-29 sum (Uh Hl + Ul Hh): three mad.wide a product.
//    The dropped 2^-58 Ul Hl is below 1/4 unit and has zero mean;
//  * the eight directions accumulate in 64-bit integers at the largest of
//    their eight exponents, to which each projected vector is rounded.  Bound:
//    reals below 2^57 units, |h| <= sqrt(3) 2 sqrt(2) 2^57 for a projected
//    colour vector, |U h| = |h|, eight directions: below 2^62.3.
//
// The result is rounded to FP64 once.  Error of a real: at most 96 units (per
// direction 4.9 from the reals, which are off by half a unit, or one where they
// are smaller than that; 1.2 from the alignment, 2.8 from the low products, 3
// from the links; 3 units rms in all), which relative to the neighbours'
// largest real is below that of FP64 sums.  But a real can be made of small
// terms alone (a colour or a spin that is small all over the neighbourhood,
// links that hardly mix colours), and FP64 keeps its 53 bits.  So the sums are
// taken only where each of them has a term U h of at least 2^-kFxSmall of the
// unit's 2^56 in it, or nothing but exact zeros (hop_terms): then the error is
// at most 96 2^-51 of the largest term (3 2^-51 rms).  Other sites, and those
// with a neighbour of Inf, NaN or extreme magnitude (exponent field of the
// largest real outside [64, 2030]: E = kFxRaw), are computed again in FP64
// from the doubles behind the integers and from the links as they are stored
// (hop_fp64).  Where the eight terms are alike in size, one real in 2^37 finds
// all of them small.
//
// Measured, a half of S at 16^4, Ls = 16 with its input pass (524288 5D sites):
// FP64 arithmetic 0.90 to 1.15 ms (FP64 pipe 88-90% busy), this form 0.28 to
// 0.31 ms.  Error of K, K^dag and H against extended precision (random SU(3),
// Ls 4 to 16): 1.61e-16 to 1.69e-16 relative, 1.66e-16 to 1.99e-16 with FP64
// arithmetic.
#pragma once

#include "common.cuh"

namespace eofa {

typedef long long i64;

constexpr int kFxFrac = 56;  // fraction bits below the block exponent
constexpr int kFxLimb = 29;  // bits of a low limb

// a 58-bit fixed-point value as its two limbs
__device__ __forceinline__ int2 fx_split(i64 v) {
    const int lo = ((int)v << 3) >> 3;  // low 29 bits, signed
    return make_int2((int)((v + (1 << (kFxLimb - 1))) >> kFxLimb), lo);
}

// the double (hi, lo) in units of 2^(E - 1023 - frac), rounded, but 1 or -1
// where that would make 0 of another number; E at least its exponent field and
// 64, frac 56 (spinors) or 58 (links)
template <int FRAC>
__device__ __forceinline__ i64 fx_from(int hi, unsigned lo, int E) {
    const unsigned mh = ((unsigned)hi & 0xfffffu) | (((unsigned)hi & 0x7fffffffu) | lo ? 0x100000u : 0u);
    const int sh = min(E - (int)(((unsigned)hi >> 20) & 0x7ffu), FRAC + 1);
    const i64 m = (i64)((((((unsigned long long)mh << 32) | lo) << (FRAC - 51) >> sh) + 1) >> 1);
    return hi < 0 ? -m : m;
}

// a link real (|u| <= 1 + 1e-10) as 58-bit fixed point
__device__ __forceinline__ i64 fx_link(double u) {
    return fx_from<2 * kFxLimb>(__double2hiint(u), (unsigned)__double2loint(u), 1023);
}

constexpr int kFxRaw = 2047;     // exponent mark of a spinor that has no integer form
constexpr int kFxSmall = 5;      // a term below 2^-5 of the unit's 2^56 is small

// N reals of a spinor -> their fixed-point form; returns E (0 for a zero
// spinor, kFxRaw for one that has no such form).  N = 12: the two lanes (sp = 0, 1) of a spinor share its exponent;
// mask: the lanes that call.
template <int N>
__device__ __forceinline__ int fx_pack(const double* v, i64* m, unsigned mask = 0) {
    int top = 0;
    unsigned low = 0;
#pragma unroll
    for (int i = 0; i < N; ++i) {
        top = max(top, __double2hiint(v[i]) & 0x7fffffff);
        low |= (unsigned)__double2loint(v[i]);
    }
    if constexpr (N == 12) {
        top = max(top, __shfl_xor_sync(mask, top, 1));
        low |= __shfl_xor_sync(mask, low, 1);
    }
    const int E = top >> 20;
    if (E < 64 || E > 2030) {
        const bool zero = top == 0 && low == 0;
#pragma unroll
        for (int i = 0; i < N; ++i) m[i] = 0;
        return zero ? 0 : kFxRaw;
    }
#pragma unroll
    for (int i = 0; i < N; ++i) m[i] = fx_from<kFxFrac>(__double2hiint(v[i]), (unsigned)__double2loint(v[i]), E);
    return E;
}

// the fixed-point spinor of 5D site (xcb, s), its exponent in the site's scale slot
__device__ __forceinline__ void fx_store(void* base, float* nrm, long xcb, int s, int Ls, const double* v) {
    i64 m[24];
    const int E = fx_pack<24>(v, m);
    longlong2* p = reinterpret_cast<longlong2*>(base) + xcb * 12 * Ls + s;
#pragma unroll
    for (int c = 0; c < 12; ++c) p[c * Ls] = make_longlong2(m[2 * c], m[2 * c + 1]);
    reinterpret_cast<int*>(nrm)[xcb * Ls + s] = E;
}

// units of 2^(E - 1023 - 56) -> double, E in [64, 2030] unless v = 0
__device__ __forceinline__ double fx_to(i64 v, int E) {
    const double d = (double)v;  // |v| < 2^63: rounded to nearest
    const int hi = __double2hiint(d) + ((E - 1023 - kFxFrac) << 20);
    return v == 0 ? 0.0 : __hiloint2double(hi, __double2loint(d));
}

// a b + c.  With (i64)a * b + c in its place H at 24^3x64, Ls = 12 takes 11.1
// instead of 7.2 ms, K at 16^4, Ls = 16 905 instead of 608 us.
__device__ __forceinline__ i64 fx_mad(int a, int b, i64 c) {
    i64 d;
    asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(d) : "r"(a), "r"(b), "l"(c));
    return d;
}

// a link element: x, y the limbs of the real part, z, w of the imaginary part
__device__ __forceinline__ int4 fx_elem(i64 re, i64 im) {
    const int2 r = fx_split(re), i = fx_split(im);
    return make_int4(r.x, r.y, i.x, i.y);
}

// rows 0 and 1 of a link (12 doubles) -> the 9 elements of W, the link or
// (dag) its adjoint; row 2 = conj(row 0 x row 1) in fixed point; neg: the
// hop's boundary sign
__device__ __forceinline__ void fx_stage_link(const double* u, bool neg, bool dag, int4* dst) {
    int4 e[9];
#pragma unroll
    for (int i = 0; i < 6; ++i) e[i] = fx_elem(fx_link(u[2 * i]), fx_link(u[2 * i + 1]));
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        const int4 a = e[(j + 1) % 3], b = e[3 + (j + 2) % 3], c = e[(j + 2) % 3], d = e[3 + (j + 1) % 3];
        // re(a b - c d) and -im(a b - c d)
        i64 rh = 0, rm = 1 << (kFxLimb - 1), ih = 0, im = 1 << (kFxLimb - 1);
        auto acc = [](int xh, int xl, int yh, int yl, i64& h, i64& m) {
            h = fx_mad(xh, yh, h);
            m = fx_mad(xh, yl, m);
            m = fx_mad(xl, yh, m);
        };
        acc(a.x, a.y, b.x, b.y, rh, rm);
        acc(a.z, a.w, -b.z, -b.w, rh, rm);
        acc(c.x, c.y, -d.x, -d.y, rh, rm);
        acc(c.z, c.w, d.z, d.w, rh, rm);
        acc(a.x, a.y, -b.z, -b.w, ih, im);
        acc(a.z, a.w, -b.x, -b.y, ih, im);
        acc(c.x, c.y, d.z, d.w, ih, im);
        acc(c.z, c.w, d.x, d.y, ih, im);
        e[6 + j] = fx_elem(rh + (rm >> kFxLimb), ih + (im >> kFxLimb));
    }
    const int sr = neg ? -1 : 1, si = neg != dag ? -1 : 1;
#pragma unroll
    for (int i = 0; i < 9; ++i)
        dst[dag ? (i % 3) * 3 + i / 3 : i] = make_int4(sr * e[i].x, sr * e[i].y, si * e[i].z, si * e[i].w);
}

// lane sp's share of a packed spinor: spins sp and 2 + sp (N = 12 reals)
__device__ __forceinline__ void fx_store_part(void* base, float* nrm, long xcb, int s, int Ls, int sp, const double* v,
                                              unsigned mask) {
    i64 m[12];
    const int E = fx_pack<12>(v, m, mask);
    longlong2* p = reinterpret_cast<longlong2*>(base) + (xcb * 12 + 3 * sp) * Ls + s;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        p[c * Ls] = make_longlong2(m[2 * c], m[2 * c + 1]);
        p[(6 + c) * Ls] = make_longlong2(m[6 + 2 * c], m[6 + 2 * c + 1]);
    }
    if (sp == 0) reinterpret_cast<int*>(nrm)[xcb * Ls + s] = E;
}

// w = W h for one colour vector, W the staged link (already daggered for a
// backward hop)
__device__ __forceinline__ void fx_mul(const int4* __restrict__ W, const i64* __restrict__ h, i64* __restrict__ w) {
    int2 hr[3], hi[3], hn[3];  // limbs of re, im and -im
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        hr[c] = fx_split(h[2 * c]);
        hi[c] = fx_split(h[2 * c + 1]);
        hn[c] = make_int2(-hi[c].x, -hi[c].y);
    }
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        // high products, and the two kinds of middle products (the first from 1/2)
        i64 Hr = 0, Hi = 0, Mr = 1 << (kFxLimb - 1), Mi = 1 << (kFxLimb - 1), Nr = 0, Ni = 0;
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            const int4 e = W[a * 3 + b];
            Hr = fx_mad(e.x, hr[b].x, Hr);
            Hi = fx_mad(e.x, hi[b].x, Hi);
            Mr = fx_mad(e.x, hr[b].y, Mr);
            Mi = fx_mad(e.x, hi[b].y, Mi);
            Nr = fx_mad(e.y, hr[b].x, Nr);
            Ni = fx_mad(e.y, hi[b].x, Ni);
            Hr = fx_mad(e.z, hn[b].x, Hr);
            Hi = fx_mad(e.z, hr[b].x, Hi);
            Mr = fx_mad(e.z, hn[b].y, Mr);
            Mi = fx_mad(e.z, hr[b].y, Mi);
            Nr = fx_mad(e.w, hn[b].x, Nr);
            Ni = fx_mad(e.w, hr[b].x, Ni);
        }
        w[2 * a] = Hr + ((Mr + Nr) >> kFxLimb);
        w[2 * a + 1] = Hi + ((Mi + Ni) >> kFxLimb);
    }
}

}  // namespace eofa
