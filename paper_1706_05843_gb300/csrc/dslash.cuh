// dslash.cuh -- the fused 4D Wilson hop + fifth-dimension kernel.
//
// One CTA owns NS output 4D sites of one checkerboard parity and all Ls
// slices of them; thread (i, s) owns 5D site (x_i, s).  Three phases:
//
//  1. hop:   h(x, s) = sum_mu [ (1 - g gamma_mu) U_mu(x) chi(x+mu, s)
//                             + (1 + g gamma_mu) U_mu(x-mu)^dag chi(x-mu, s) ]
//            with g = +1 (D_h) or -1 (gamma_5 D_h gamma_5 = the hop of D^dag),
//            chi = psi, or chi = D~ psi / b5 built on the fly from the
//            neighbour's slices s-1 (P+ half) and s+1 (P- half) -- the
//            "L acts first" order of Eq. (Ddwf).  Spin projection to half
//            spinors, two-row links rebuilt in registers; h goes to shared
//            memory.  An optional site-local input y is staged beside it.
//            FP64: the products run in 64-bit fixed point on inputs prepared
//            for it, and in FP64 where a sum needs that (fixed64.cuh), two
//            lanes to a 5D site; a pass over the input applies D~ where a
//            kind wants it.
//  2. fifth dimension: each thread takes complex columns (x_i, spin, colour)
//            and applies an O(Ls) program: the cyclic bidiagonal
//            A = alpha + gamma L (the site-diagonal block of D_DWF, App. B),
//            its transpose, its inverse by a closed-form corner plus a
//            first-order recurrence, the rank-one EOFA shift u (x) v
//            (Eqs. Mooee_shift_p/m) and its Sherman-Morrison inverse
//            (Eq. sherman_morrison_mobius_inv), D~ = b5 + c5 L and D~^T.
//            The site-local kinds (M y + h: L reaches one neighbouring
//            slice, the shift one fixed slice) skip this phase: thread
//            (i, s) reads those slices of y itself and keeps h in registers.
//  3. store: thread (i, s) writes its spinor back (coalesced 16-byte
//            chunks) and contributes |out|^2 to a deterministic reduction.
//
// The kernel kinds below are the even-odd blocks of K (App. B):
//   K_ee = K_oo = M (site-local), K_eo = K_oe = -1/2 D_h D~,
// and of K D~^-1, which the inner CG inverts.
#pragma once

#include <type_traits>

#include "common.cuh"
#include "fixed64.cuh"

namespace eofa {

enum Kind {
    KIND_EO_MINV = 0,      // out = -1/2 D~ M^-1 D_h D~ in            (Schur step 1)
    KIND_OE_SCHUR = 1,     // out = M y + 1/2 D_h in                  (Schur step 2; in = D~ t)
    KIND_EO_MINV_DAG = 2,  // out = -1/2 M^-T D~^T g5 D_h g5 in       (Schur^dag step 1)
    KIND_OE_SCHUR_DAG = 3, // out = M^T y + 1/2 D~^T g5 D_h g5 in     (Schur^dag step 2)
    KIND_RECON = 4,        // out = M^-1 (y + 1/2 D_h D~ in)          (even reconstruction)
    KIND_SRC = 5,          // out = y + 1/2 D_h in                    (even-odd source)
    KIND_FULL = 6,         // out = M y - 1/2 D_h D~ in               (K, one parity)
    KIND_FULL_DAG = 7,     // out = M^T y - 1/2 D~^T g5 D_h g5 in     (K^dag, one parity)
    KIND_LOC_DTMINV = 8,   // out = D~ M^-1 y
    KIND_LOC_DT = 9,       // out = D~ y
    KIND_LOC_DTINV = 10,   // out = D~^-1 y
    // even-odd on Eq. (non_hermit_sys) without the Cayley form (App. B):
    // A = D_EOFA + beta g5 R5 Delta P, A_ee = A_oo dense in s, A_eo = -1/2 D_h
    KIND_D_EO = 11,        // out = -1/2 A_ee^-1 D_h in
    KIND_D_OE = 12,        // out = A_oo y + 1/2 D_h in
    KIND_D_EO_DAG = 13,    // out = -1/2 A_ee^-T g5 D_h g5 in
    KIND_D_OE_DAG = 14,    // out = A_oo^T y + 1/2 g5 D_h g5 in
    // the inner operator of the Cayley-form solve, kT S D~^-1 (App. B's scheme
    // with the right preconditioner taken out again inside the CG): with
    // T = D~ M^-1, kT = b5 / alpha and h = D_h in or g5 D_h g5 in
    KIND_R_EO = 15,        // out = T h / kT
    KIND_R_OE = 16,        // out = kT T^-1 y - kT^2 / 4 h
    KIND_R_EO_DAG = 17,    // out = T^T h / kT
    KIND_R_OE_DAG = 18,    // out = kT T^-T y - kT^2 / 4 h
    KIND_R_BACK = 19,      // out = kT D~^-1 y
    KIND_H = 20,           // out = T^-1 y - 1/2 D_h y = K D~^-1 y, one parity (in = y; FP64)
    NKIND = 21
};

template <int K> struct KindTraits {
    static constexpr bool DENSE = K >= KIND_D_EO && K <= KIND_D_OE_DAG;
    static constexpr bool HOP = K <= KIND_FULL_DAG || DENSE || (K >= KIND_R_EO && K <= KIND_R_OE_DAG) || K == KIND_H;
    static constexpr bool DAG = K == KIND_EO_MINV_DAG || K == KIND_OE_SCHUR_DAG || K == KIND_FULL_DAG ||
                                K == KIND_D_EO_DAG || K == KIND_D_OE_DAG || K == KIND_R_EO_DAG || K == KIND_R_OE_DAG;
    static constexpr bool PRE = K == KIND_EO_MINV || K == KIND_RECON || K == KIND_FULL;
    static constexpr bool HASY = !(K == KIND_EO_MINV || K == KIND_EO_MINV_DAG || K == KIND_D_EO || K == KIND_D_EO_DAG ||
                                   K == KIND_R_EO || K == KIND_R_EO_DAG);
    // the column program acts on y alone and runs before the hop, whose
    // result stays in registers: one staged tile instead of two
    static constexpr bool YCOL = K == KIND_R_OE || K == KIND_R_OE_DAG || K == KIND_H;
    // the operator applications: y and out may be the caller's canonical fields
    static constexpr bool APPLY = K == KIND_FULL || K == KIND_FULL_DAG || K == KIND_H;
    // FP64: the output is only ever the hop input of the next kernel and is
    // stored in its fixed-point form (fixed64.cuh), its doubles beside it
    static constexpr bool FXOUT = K == KIND_EO_MINV || K == KIND_EO_MINV_DAG || K == KIND_D_EO ||
                                  K == KIND_D_EO_DAG || K == KIND_LOC_DTMINV || K == KIND_R_EO || K == KIND_R_EO_DAG;
    // site-local kinds: the fifth-dimension part reaches only slices s-1, s+1
    // and the fixed slice of the rank-one shift, so each thread finishes its
    // own 5D site without the shared-memory column phase
    static constexpr bool PTW = K == KIND_OE_SCHUR || K == KIND_SRC || K == KIND_FULL;
};

struct HopArgs {
    Geom g;
    int out_par;
    int tile_var;                            // CTA tile variant (autotuner)
    const void* in;  const float* in_nrm;    // hop input, parity 1 - out_par (FP64: fixed point, exponents in in_nrm)
    const void* in_raw;                      // FP64: the field that the hop input was made from (without D~)
    const void* y;   const float* y_nrm;     // site-local input, parity out_par
    void* out;       float* out_nrm;         // output, parity out_par
    void* out_raw;                           // KT::FXOUT: the output's doubles beside its fixed-point form
    const void* lk_out;                      // links of parity out_par
    const void* lk_in;                       // links of parity 1 - out_par
    Reduce rd;                               // rd.fin == FIN_NONE: no reduction
    const int* done;                         // early exit when *done != 0 (may be NULL)
    int* stop;                               // set by a launch that finds *done set (may be NULL)
    int prepare;                             // 1: set the kernel up on the current device, launch nothing
    int canon;                               // KT::APPLY kinds, bit 0: y, in_raw and out are canonical complex128
                                             // fields of the whole lattice; bit 1: out takes gamma_5 R_5
    // dense kinds: the Ls x Ls s-space matrix of each chirality in compute
    // precision, [chirality][row][col] in mirrored coordinates
    // (A_ee^-1 for the EO kinds, A_oo for the OE kinds)
    const void* dense;
};

// ---------------------------------------------------------------------------
// complex helpers
// ---------------------------------------------------------------------------
template <typename R> struct C2 { R re, im; };

template <typename R>
__device__ __forceinline__ C2<R> cmul(C2<R> a, C2<R> b) {
    return {a.re * b.re - a.im * b.im, a.re * b.im + a.im * b.re};
}
template <typename R>
__device__ __forceinline__ C2<R> cmulc(C2<R> a, C2<R> b) {  // conj(a) * b
    return {a.re * b.re + a.im * b.im, a.re * b.im - a.im * b.re};
}

// ---------------------------------------------------------------------------
// one hopping direction: acc += (1 + SG gamma_MU) W chi, W = U or U^dag
// u: 18 reals, rows 0..2 of the link (row 2 rebuilt; the boundary sign of the
// hop folded in).
// ---------------------------------------------------------------------------
template <typename R, int MU, int SG, bool ADJ>
__device__ __forceinline__ void hop_dir(R* __restrict__ acc, const R* __restrict__ p,
                                        const R* __restrict__ u) {
    // spin projection: h = psi_up + SG B psi_dn, B = -i sigma_k (k = 1..3) or 1
    R h[12];
    constexpr R s = (R)SG;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const R p0r = p[0 * 6 + 2 * c], p0i = p[0 * 6 + 2 * c + 1];
        const R p1r = p[1 * 6 + 2 * c], p1i = p[1 * 6 + 2 * c + 1];
        const R p2r = p[2 * 6 + 2 * c], p2i = p[2 * 6 + 2 * c + 1];
        const R p3r = p[3 * 6 + 2 * c], p3i = p[3 * 6 + 2 * c + 1];
        R h0r, h0i, h1r, h1i;
        if constexpr (MU == 0) {        // B psi_dn = (-i psi3, -i psi2)
            h0r = p0r + s * p3i; h0i = p0i - s * p3r;
            h1r = p1r + s * p2i; h1i = p1i - s * p2r;
        } else if constexpr (MU == 1) { // B psi_dn = (-psi3, psi2)
            h0r = p0r - s * p3r; h0i = p0i - s * p3i;
            h1r = p1r + s * p2r; h1i = p1i + s * p2i;
        } else if constexpr (MU == 2) { // B psi_dn = (-i psi2, i psi3)
            h0r = p0r + s * p2i; h0i = p0i - s * p2r;
            h1r = p1r - s * p3i; h1i = p1i + s * p3r;
        } else {                        // B psi_dn = psi_dn
            h0r = p0r + s * p2r; h0i = p0i + s * p2i;
            h1r = p1r + s * p3r; h1i = p1i + s * p3i;
        }
        h[2 * c] = h0r; h[2 * c + 1] = h0i;
        h[6 + 2 * c] = h1r; h[6 + 2 * c + 1] = h1i;
    }
    // colour: w = W h for both half-spinor components
    R w[12];
#pragma unroll
    for (int sp = 0; sp < 2; ++sp) {
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            // complex multiply-accumulate as plain FMA chains (4 per term)
            R re = (R)0, im = (R)0;
#pragma unroll
            for (int b = 0; b < 3; ++b) {
                const R hr = h[sp * 6 + 2 * b], hi = h[sp * 6 + 2 * b + 1];
                if constexpr (!ADJ) {       // U_ab h_b
                    const R ur = u[(a * 3 + b) * 2], ui = u[(a * 3 + b) * 2 + 1];
                    if (b == 0) { re = ur * hr; im = ur * hi; }
                    else { re = fma(ur, hr, re); im = fma(ur, hi, im); }
                    re = fma(-ui, hi, re);
                    im = fma(ui, hr, im);
                } else {                    // conj(U_ba) h_b
                    const R ur = u[(b * 3 + a) * 2], ui = u[(b * 3 + a) * 2 + 1];
                    if (b == 0) { re = ur * hr; im = ur * hi; }
                    else { re = fma(ur, hr, re); im = fma(ur, hi, im); }
                    re = fma(ui, hi, re);
                    im = fma(-ui, hr, im);
                }
            }
            w[sp * 6 + 2 * a] = re;
            w[sp * 6 + 2 * a + 1] = im;
        }
    }
    // reconstruct: upper += w, lower += SG B^dag w
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const R w0r = w[2 * c], w0i = w[2 * c + 1];
        const R w1r = w[6 + 2 * c], w1i = w[6 + 2 * c + 1];
        acc[0 * 6 + 2 * c] += w0r; acc[0 * 6 + 2 * c + 1] += w0i;
        acc[1 * 6 + 2 * c] += w1r; acc[1 * 6 + 2 * c + 1] += w1i;
        if constexpr (MU == 0) {        // B^dag w = (i w1, i w0)
            acc[2 * 6 + 2 * c] -= s * w1i; acc[2 * 6 + 2 * c + 1] += s * w1r;
            acc[3 * 6 + 2 * c] -= s * w0i; acc[3 * 6 + 2 * c + 1] += s * w0r;
        } else if constexpr (MU == 1) { // B^dag w = (w1, -w0)
            acc[2 * 6 + 2 * c] += s * w1r; acc[2 * 6 + 2 * c + 1] += s * w1i;
            acc[3 * 6 + 2 * c] -= s * w0r; acc[3 * 6 + 2 * c + 1] -= s * w0i;
        } else if constexpr (MU == 2) { // B^dag w = (i w0, -i w1)
            acc[2 * 6 + 2 * c] -= s * w0i; acc[2 * 6 + 2 * c + 1] += s * w0r;
            acc[3 * 6 + 2 * c] += s * w1i; acc[3 * 6 + 2 * c + 1] -= s * w1r;
        } else {                        // B^dag w = w
            acc[2 * 6 + 2 * c] += s * w0r; acc[2 * 6 + 2 * c + 1] += s * w0i;
            acc[3 * 6 + 2 * c] += s * w1r; acc[3 * 6 + 2 * c + 1] += s * w1i;
        }
    }
}

template <typename R>
__device__ __forceinline__ void rebuild_row2(R* u) {
    // row2 = conj(row0 x row1)
    C2<R> a0 = {u[0], u[1]}, a1 = {u[2], u[3]}, a2 = {u[4], u[5]};
    C2<R> b0 = {u[6], u[7]}, b1 = {u[8], u[9]}, b2 = {u[10], u[11]};
    C2<R> c0 = cmul(a1, b2), d0 = cmul(a2, b1);
    C2<R> c1 = cmul(a2, b0), d1 = cmul(a0, b2);
    C2<R> c2 = cmul(a0, b1), d2 = cmul(a1, b0);
    u[12] = c0.re - d0.re; u[13] = -(c0.im - d0.im);
    u[14] = c1.re - d1.re; u[15] = -(c1.im - d1.im);
    u[16] = c2.re - d2.re; u[17] = -(c2.im - d2.im);
}

// ---------------------------------------------------------------------------
// fifth-dimension column operators (mirrored coordinates: always L+ / L-)
// ---------------------------------------------------------------------------
// A column holds one value per slice: a complex number for FP32 arithmetic, a
// real one for FP64 (every coefficient is real), so that the few sites of an
// FP64 tile still give 24 columns each.
template <typename R> struct C1 { R re; };
template <typename R> struct ColVal { typedef C2<R> V; };
template <> struct ColVal<double> { typedef C1<double> V; };

template <typename R> __device__ __forceinline__ C2<R> vmul(R a, C2<R> x) { return {a * x.re, a * x.im}; }
template <typename R> __device__ __forceinline__ C1<R> vmul(R a, C1<R> x) { return {a * x.re}; }
// a x + y
template <typename R> __device__ __forceinline__ C2<R> vfma(R a, C2<R> x, C2<R> y) {
    return {fma(a, x.re, y.re), fma(a, x.im, y.im)};
}
template <typename R> __device__ __forceinline__ C1<R> vfma(R a, C1<R> x, C1<R> y) { return {fma(a, x.re, y.re)}; }

// (a + g L+) v,  L+: v_s <- v_{s-1}, v_0 <- -m v_{Ls-1}
template <typename R, int LS, typename V>
__device__ __forceinline__ void op_fwd(V* v, R a, R g, R mg) {
    const V last = v[LS - 1];
#pragma unroll
    for (int s = LS - 1; s >= 1; --s) v[s] = vfma(a, v[s], vmul(g, v[s - 1]));
    v[0] = vfma(a, v[0], vmul(-mg, last));
}
// (a + g L-) v = (a + g L+^T) v
template <typename R, int LS, typename V>
__device__ __forceinline__ void op_fwdT(V* v, R a, R g, R mg) {
    const V first = v[0];
#pragma unroll
    for (int s = 0; s < LS - 1; ++s) v[s] = vfma(a, v[s], vmul(g, v[s + 1]));
    v[LS - 1] = vfma(a, v[LS - 1], vmul(-mg, first));
}
// v += f a (a a vector in s, f a column value)
template <typename R, int LS, typename V>
__device__ __forceinline__ void op_axpy(V* v, const R* a, V f) {
#pragma unroll
    for (int s = 0; s < LS; ++s) v[s] = vfma(a[s], f, v[s]);
}
template <typename R, int LS, typename V>
__device__ __forceinline__ V op_dot(const V* v, const R* a) {
    V d = {};
#pragma unroll
    for (int s = 0; s < LS; ++s) d = vfma(a[s], v[s], d);
    return d;
}
// sum_j w_j v_{Ls-1-j}
template <typename R, int LS, typename V>
__device__ __forceinline__ V op_rdot(const V* v, const R* w) {
    V d = {};
#pragma unroll
    for (int j = 0; j < LS; ++j) d = vfma(w[j], v[LS - 1 - j], d);
    return d;
}
// solve (a + g L+) t = v in place: t_{Ls-1} = sum_j w_j v_{Ls-1-j},
// t_0 = v_0/a + m z t_{Ls-1}, t_s = v_s/a - z t_{s-1}.
template <typename R, int LS, typename V>
__device__ __forceinline__ void op_inv(V* v, R ia, R z, R mz, const R* w) {
    const V tl = op_rdot<R, LS>(v, w);
    v[0] = vfma(ia, v[0], vmul(mz, tl));
#pragma unroll
    for (int s = 1; s < LS - 1; ++s) v[s] = vfma(ia, v[s], vmul(-z, v[s - 1]));
    v[LS - 1] = tl;
}
// solve (a + g L-) t = v in place (the mirror image of op_inv)
template <typename R, int LS, typename V>
__device__ __forceinline__ void op_invT(V* v, R ia, R z, R mz, const R* w) {
    const V t0 = op_dot<R, LS>(v, w);
    v[LS - 1] = vfma(ia, v[LS - 1], vmul(mz, t0));
#pragma unroll
    for (int s = LS - 2; s >= 1; --s) v[s] = vfma(ia, v[s], vmul(-z, v[s + 1]));
    v[0] = t0;
}

// M = A + pm beta u (x) v  on the shift chirality
template <typename R, int LS, typename V>
__device__ __forceinline__ void op_M(V* v, const SCoef<R>& c, bool sh) {
    const V vl = v[LS - 1];
    op_fwd<R, LS>(v, c.alpha, c.gamma, c.m * c.gamma);
    if (sh) op_axpy<R, LS>(v, c.um, vmul(c.sbk, vl));
}
template <typename R, int LS, typename V>
__device__ __forceinline__ void op_MT(V* v, const SCoef<R>& c, bool sh) {
    V d = {};
    if (sh) d = op_dot<R, LS>(v, c.um);
    op_fwdT<R, LS>(v, c.alpha, c.gamma, c.m * c.gamma);
    if (sh) v[LS - 1] = vfma(c.sbk, d, v[LS - 1]);
}
// Sherman-Morrison: M^-1 v = A^-1 v - (pm beta k (A^-1 v)_{j*} / den) x
template <typename R, int LS, typename V>
__device__ __forceinline__ void op_Minv(V* v, const SCoef<R>& c, bool sh) {
    op_inv<R, LS>(v, c.ia, c.za, c.mza, c.wa);
    if (sh) op_axpy<R, LS>(v, c.xm, vmul(-c.sbk_den, v[LS - 1]));
}
// M^-T v = A^-T v - (pm beta (u . A^-T v) / den) y
template <typename R, int LS, typename V>
__device__ __forceinline__ void op_MinvT(V* v, const SCoef<R>& c, bool sh) {
    op_invT<R, LS>(v, c.ia, c.za, c.mza, c.wa);
    if (sh) op_axpy<R, LS>(v, c.ym, vmul(-c.sb_den, op_dot<R, LS>(v, c.um)));
}

// The factors of the right-preconditioned inner operator (3.5 to 4.5
// multiply-adds per real instead of 6.5 for D~ M^-1 done in two recurrences;
// 16^4, Ls = 16, one launch: FP64 0.31 -> 0.24 ms, FP32 without the D~ pre-op
// 0.050 -> 0.038 ms for the first half, 0.042 ms for the second).  With a cyclic
// bidiagonal Z = 1 + z L and v = Z q, one recurrence gives L q beside q:
// (L q)_0 = -m q_last, q_s = v_s - z (L q)_s, (L q)_{s+1} = q_s.
// v <- v + g L q;  returns q_last = sum_j w_j v_{Ls-1-j}
template <typename R, int LS, typename V>
__device__ __forceinline__ V op_pade(V* v, R z, R g, R m, const R* w) {
    const V last = op_rdot<R, LS>(v, w);
    V l = vmul(-m, last);
#pragma unroll
    for (int s = 0; s < LS; ++s) {
        const V q = vfma(-z, l, v[s]);
        v[s] = vfma(g, l, v[s]);
        l = q;
    }
    return last;
}
// the transpose: Z = 1 + z L^T, v <- v + g L^T q
template <typename R, int LS, typename V>
__device__ __forceinline__ void op_padeT(V* v, R z, R g, R m, const R* w) {
    V l = vmul(-m, op_dot<R, LS>(v, w));
#pragma unroll
    for (int s = LS - 1; s >= 0; --s) {
        const V q = vfma(-z, l, v[s]);
        v[s] = vfma(g, l, v[s]);
        l = q;
    }
}

// ---------------------------------------------------------------------------
// shared-memory staging of the 5D tile
// ---------------------------------------------------------------------------
// A tile row holds the 24 reals of one 5D site.  The P- half (spins 2, 3) of
// slice s is stored in row Ls-1-s, so a column of either chirality reads its
// mirrored coordinate (the one in which both L's are L+) in row order.
template <typename R> struct ShStride;
template <> struct ShStride<float> { static constexpr int V = 28; };   // 112 B rows: conflict-free float4
template <> struct ShStride<double> { static constexpr int V = 26; };  // 208 B rows: conflict-free double2

// rows of one 4D site, padded so that the 12 columns of consecutive sites
// land on consecutive (re, im) bank pairs of a 128-byte line
template <typename R, int LS> struct SiteStride {
    static constexpr int MOD = 128 / (int)sizeof(R);
    static constexpr int WANT = 24 % MOD;
    static constexpr int V = LS * ShStride<R>::V + ((WANT - (LS * ShStride<R>::V) % MOD) + MOD) % MOD;
};

template <typename R> struct Pair;
template <> struct Pair<float> { typedef float2 T; };
template <> struct Pair<double> { typedef double2 T; };
template <typename R> struct Quad;
template <> struct Quad<float> { typedef float4 T; static constexpr int N = 4; };
template <> struct Quad<double> { typedef double2 T; static constexpr int N = 2; };

template <typename R>
__device__ __forceinline__ C2<R> ld_pair(const R* p) {
    const typename Pair<R>::T q = *reinterpret_cast<const typename Pair<R>::T*>(p);
    return {q.x, q.y};
}
template <typename R>
__device__ __forceinline__ void st_pair(R* p, const C2<R>& v) {
    typename Pair<R>::T q;
    q.x = v.re;
    q.y = v.im;
    *reinterpret_cast<typename Pair<R>::T*>(p) = q;
}
// M reals (one chirality half of a row, or a lane's part of it) as 16-byte vectors
template <int M, typename R>
__device__ __forceinline__ void st_half(R* p, const R* v) {
    typedef typename Quad<R>::T Q;
    constexpr int N = Quad<R>::N;
#pragma unroll
    for (int i = 0; i < M / N; ++i) {
        Q q;
        if constexpr (N == 4) q = make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
        else q = make_double2(v[2 * i], v[2 * i + 1]);
        reinterpret_cast<Q*>(p)[i] = q;
    }
}
template <int M, typename R>
__device__ __forceinline__ void ld_half(const R* p, R* v) {
    typedef typename Quad<R>::T Q;
    constexpr int N = Quad<R>::N;
#pragma unroll
    for (int i = 0; i < M / N; ++i) {
        const Q q = reinterpret_cast<const Q*>(p)[i];
        if constexpr (N == 4) {
            v[4 * i] = q.x; v[4 * i + 1] = q.y; v[4 * i + 2] = q.z; v[4 * i + 3] = q.w;
        } else {
            v[2 * i] = q.x; v[2 * i + 1] = q.y;
        }
    }
}

// Column access of a shared tile: one value per row, rows ST reals apart.
template <typename R, int LS, int ST>
__device__ __forceinline__ void col_load(const R* p, C2<R>* v) {
#pragma unroll
    for (int k = 0; k < LS; ++k) v[k] = ld_pair(p + k * ST);
}
template <typename R, int LS, int ST>
__device__ __forceinline__ void col_load(const R* p, C1<R>* v) {
#pragma unroll
    for (int k = 0; k < LS; ++k) v[k] = {p[k * ST]};
}
template <typename R, int LS, int ST>
__device__ __forceinline__ void col_store(R* p, const C2<R>* v) {
#pragma unroll
    for (int k = 0; k < LS; ++k) st_pair(p + k * ST, v[k]);
}
template <typename R, int LS, int ST>
__device__ __forceinline__ void col_store(R* p, const C1<R>* v) {
#pragma unroll
    for (int k = 0; k < LS; ++k) p[k * ST] = v[k].re;
}

// The fifth-dimension program of one (site, spin, colour) column (of its real
// or imaginary part for FP64), in the mirrored coordinate.  hcol: the hop
// result (overwritten with the output), ycol: the local input; consecutive
// slices are ST reals apart.
template <typename R, int LS, int KIND, int ST>
__device__ __forceinline__ void column_program(R* hcol, const R* ycol, const SCoef<R>& cf, bool shv,
                                               R hb, const R* mat) {
    typedef KindTraits<KIND> KT;
    typedef typename ColVal<R>::V V;
    V v[LS];
    if constexpr (KT::DENSE) {
        // dense s-space matrix (row-major in mirrored coordinates) times the
        // column, or its transpose for the adjoint kinds
        constexpr bool TR = KT::DAG;
        constexpr bool EO = (KIND == KIND_D_EO || KIND == KIND_D_EO_DAG);
        col_load<R, LS, ST>(EO ? hcol : ycol, v);
        V w[LS];
#pragma unroll
        for (int k = 0; k < LS; ++k) {
            w[k] = {};
#pragma unroll
            for (int j = 0; j < LS; ++j) w[k] = vfma(TR ? mat[j * LS + k] : mat[k * LS + j], v[j], w[k]);
        }
        if constexpr (EO) {
#pragma unroll
            for (int k = 0; k < LS; ++k) v[k] = vmul((R)-0.5, w[k]);
        } else {
            V h[LS];
            col_load<R, LS, ST>(hcol, h);
#pragma unroll
            for (int k = 0; k < LS; ++k) v[k] = vfma((R)0.5, h[k], w[k]);
        }
    } else if constexpr (KIND == KIND_R_EO) {
        col_load<R, LS, ST>(hcol, v);
        const V l = op_pade<R, LS>(v, cf.za, cf.g1, cf.m, cf.wu);
        if (shv) op_axpy<R, LS>(v, cf.xD, vmul((R)-1, l));
    } else if constexpr (KIND == KIND_R_EO_DAG) {
        col_load<R, LS, ST>(hcol, v);
        op_padeT<R, LS>(v, cf.za, cf.g1, cf.m, cf.wu);
        if (shv) op_axpy<R, LS>(v, cf.yn, vmul((R)-1, op_dot<R, LS>(v, cf.um)));
    } else if constexpr (KIND == KIND_R_OE || KIND == KIND_H) {
        col_load<R, LS, ST>(hcol, v);  // the staged y
        const V l = op_pade<R, LS>(v, cf.zb, -cf.g1, cf.m, cf.wv);
        if (shv) op_axpy<R, LS>(v, cf.uT, l);
    } else if constexpr (KIND == KIND_R_OE_DAG) {
        col_load<R, LS, ST>(hcol, v);
        V d = {};
        if (shv) d = op_dot<R, LS>(v, cf.um);
        op_padeT<R, LS>(v, cf.zb, -cf.g1, cf.m, cf.wv);
        if (shv) op_axpy<R, LS>(v, cf.eD, d);
    } else if constexpr (KIND == KIND_EO_MINV) {
        col_load<R, LS, ST>(hcol, v);
        op_Minv<R, LS>(v, cf, shv);
        op_fwd<R, LS>(v, cf.b5, cf.c5, cf.m * cf.c5);
#pragma unroll
        for (int k = 0; k < LS; ++k) v[k] = vmul((R)(-0.5) * hb, v[k]);
    } else if constexpr (KIND == KIND_EO_MINV_DAG) {
        col_load<R, LS, ST>(hcol, v);
        op_fwdT<R, LS>(v, cf.b5, cf.c5, cf.m * cf.c5);
        op_MinvT<R, LS>(v, cf, shv);
#pragma unroll
        for (int k = 0; k < LS; ++k) v[k] = vmul((R)-0.5, v[k]);
    } else {
        col_load<R, LS, ST>(ycol, v);
        if constexpr (KIND == KIND_OE_SCHUR || KIND == KIND_FULL) op_M<R, LS>(v, cf, shv);
        if constexpr (KIND == KIND_OE_SCHUR_DAG || KIND == KIND_FULL_DAG) op_MT<R, LS>(v, cf, shv);
        if constexpr (KT::HOP) {
            V w[LS];
            col_load<R, LS, ST>(hcol, w);
            if constexpr (KIND == KIND_OE_SCHUR_DAG || KIND == KIND_FULL_DAG)
                op_fwdT<R, LS>(w, cf.b5, cf.c5, cf.m * cf.c5);
            const R f = ((KIND == KIND_FULL || KIND == KIND_FULL_DAG) ? (R)-0.5 : (R)0.5) * hb;
#pragma unroll
            for (int k = 0; k < LS; ++k) v[k] = vfma(f, w[k], v[k]);
        }
        if constexpr (KIND == KIND_RECON) op_Minv<R, LS>(v, cf, shv);
        if constexpr (KIND == KIND_LOC_DTMINV) {
            op_Minv<R, LS>(v, cf, shv);
            op_fwd<R, LS>(v, cf.b5, cf.c5, cf.m * cf.c5);
        }
        if constexpr (KIND == KIND_LOC_DT) op_fwd<R, LS>(v, cf.b5, cf.c5, cf.m * cf.c5);
        if constexpr (KIND == KIND_LOC_DTINV) op_inv<R, LS>(v, cf.ib, cf.zb, cf.mzb, cf.wb);
        if constexpr (KIND == KIND_R_BACK) {
            op_inv<R, LS>(v, cf.ib, cf.zb, cf.mzb, cf.wb);
#pragma unroll
            for (int k = 0; k < LS; ++k) v[k] = vmul(cf.b5 * cf.kTb, v[k]);
        }
    }
    col_store<R, LS, ST>(hcol, v);
}

// lane sp's reals of the half hi of slice s (HV = 2: spin 2 hi + sp; FP64)
template <typename S, typename R, int HV>
__device__ __forceinline__ void load_half_part(const void* __restrict__ base, const float* __restrict__ nrm, long xcb,
                                               int s, int Ls, int hi, int sp, R* v) {
    if constexpr (HV == 1) {
        load_half<S, R>(base, nrm, xcb, s, Ls, hi, v);
    } else {
        const double2* p = reinterpret_cast<const double2*>(base) + (xcb * 12 + 6 * hi + 3 * sp) * Ls + s;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const double2 t = p[c * Ls];
            v[2 * c] = t.x;
            v[2 * c + 1] = t.y;
        }
    }
}

// v <- M v for the 5D site (xcb, s) of field y, v = y(xcb, s) on entry: the
// P+ half takes slice s-1, the P- half slice s+1 (antiperiodic through -m),
// and the shift chirality the rank-one term sbk u_k y(last) of Eq. (Mooee_shift)
// with k the mirrored index and "last" slice Ls-1 (P+) or 0 (P-).
// half(s, hi, q): the half hi of slice s of y at this site.
template <typename R, int LS, int HF, typename HALF>
__device__ __forceinline__ void site_M(HALF&& half, int s, const SCoef<R>& cf, R* v) {
    R q[HF];
    {
        const int sm = (s == 0) ? LS - 1 : s - 1;
        const R gu = (s == 0) ? -cf.m * cf.gamma : cf.gamma;
        half(sm, 0, q);
#pragma unroll
        for (int i = 0; i < HF; ++i) v[i] = cf.alpha * v[i] + gu * q[i];
    }
    {
        const int sp = (s == LS - 1) ? 0 : s + 1;
        const R gd = (s == LS - 1) ? -cf.m * cf.gamma : cf.gamma;
        half(sp, 1, q);
#pragma unroll
        for (int i = 0; i < HF; ++i) v[HF + i] = cf.alpha * v[HF + i] + gd * q[i];
    }
    if (cf.has_shift) {
        const int cs = cf.cs;
        half(cs == 0 ? LS - 1 : 0, cs, q);
        const R f = cf.sbk * cf.um[cs == 0 ? s : LS - 1 - s];
        if (cs == 0) {
#pragma unroll
            for (int i = 0; i < HF; ++i) v[i] += f * q[i];
        } else {
#pragma unroll
            for (int i = 0; i < HF; ++i) v[HF + i] += f * q[i];
        }
    }
}

// The adjoint site-local kinds (M^T y + f D~^T h) need slice s+1 (P+) and
// s-1 (P-) of both y and h, and on the shift chirality the column sum
// d = sum_k u_k y_k.  When Ls is a power of two the Ls threads of a 4D site
// are one aligned lane group of a warp, and these come from warp shuffles;
// otherwise (Ls = 12) the kind goes through the column phase.
template <int K, int LS> struct ShflTail {
    static constexpr bool ON = (K == KIND_OE_SCHUR_DAG || K == KIND_FULL_DAG) && LS <= 32 && (LS & (LS - 1)) == 0;
    static constexpr bool COLS = !KindTraits<K>::PTW && !ON;
};

// o = M^T v + f (b5 + c5 L^T) h for slice s of a group of LS HV lanes (HV lanes
// a slice, 24 / HV reals each): L^T takes
// P+ from slice s+1 and P- from slice s-1, each with -m across the wall;
// the rank-one part of M^T adds sbk (sum_k u_k v_k) to the last mirrored
// slice of the shift chirality.  Every lane of the warp must call this.
template <typename R, int LS, int HV>
__device__ __forceinline__ void site_MT_dtT(int s, int sp, const SCoef<R>& cf, const R* v, const R* h, R f, R* o) {
    constexpr unsigned FULL = 0xffffffffu;
    constexpr int HF = 12 / HV, W = LS * HV;
    const int up = ((s + 1) & (LS - 1)) * HV + sp, dn = ((s - 1) & (LS - 1)) * HV + sp;
    const R wu = (s == LS - 1) ? -cf.m : (R)1;
    const R wd = (s == 0) ? -cf.m : (R)1;
    const R fb = f * cf.b5, fc = f * cf.c5;
#pragma unroll
    for (int i = 0; i < HF; ++i) {
        const R yn = wu * __shfl_sync(FULL, v[i], up, W);
        const R hn = wu * __shfl_sync(FULL, h[i], up, W);
        o[i] = cf.alpha * v[i] + cf.gamma * yn + fb * h[i] + fc * hn;
    }
#pragma unroll
    for (int i = HF; i < 2 * HF; ++i) {
        const R yn = wd * __shfl_sync(FULL, v[i], dn, W);
        const R hn = wd * __shfl_sync(FULL, h[i], dn, W);
        o[i] = cf.alpha * v[i] + cf.gamma * yn + fb * h[i] + fc * hn;
    }
    if (cf.has_shift) {
        const int cs = cf.cs;
        const R u = cf.um[cs == 0 ? s : LS - 1 - s];
        const bool last = s == (cs == 0 ? LS - 1 : 0);
        R d[HF];
        if (cs == 0) {
#pragma unroll
            for (int i = 0; i < HF; ++i) d[i] = u * v[i];
        } else {
#pragma unroll
            for (int i = 0; i < HF; ++i) d[i] = u * v[HF + i];
        }
#pragma unroll
        for (int off = LS / 2; off > 0; off >>= 1) {
#pragma unroll
            for (int i = 0; i < HF; ++i) d[i] += __shfl_xor_sync(FULL, d[i], off * HV, W);
        }
        if (last) {
            if (cs == 0) {
#pragma unroll
                for (int i = 0; i < HF; ++i) o[i] += cf.sbk * d[i];
            } else {
#pragma unroll
                for (int i = 0; i < HF; ++i) o[HF + i] += cf.sbk * d[i];
            }
        }
    }
}

// ---------------------------------------------------------------------------
// the kernel
// ---------------------------------------------------------------------------

// one staged link: 18 reals padded to a multiple of 16 bytes
template <typename R> struct LinkStride;
template <> struct LinkStride<float> { static constexpr int V = 20; };
template <> struct LinkStride<double> { static constexpr int V = 18; };

// a staged link as 16-byte shared-memory accesses (18 reals; the float
// stride of 20 keeps every link 16-byte aligned)
template <typename R>
__device__ __forceinline__ void ld_link(const R* __restrict__ src, R* u) {
    if constexpr (sizeof(R) == 4) {
        const float4* q = reinterpret_cast<const float4*>(src);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float4 t = q[i];
            u[4 * i] = t.x; u[4 * i + 1] = t.y; u[4 * i + 2] = t.z; u[4 * i + 3] = t.w;
        }
        const float2 t = reinterpret_cast<const float2*>(src)[8];
        u[16] = t.x; u[17] = t.y;
    } else {
        const double2* q = reinterpret_cast<const double2*>(src);
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            const double2 t = q[i];
            u[2 * i] = t.x; u[2 * i + 1] = t.y;
        }
    }
}
template <typename R>
__device__ __forceinline__ void st_link(R* __restrict__ dst, const R* u) {
    if constexpr (sizeof(R) == 4) {
        float4* q = reinterpret_cast<float4*>(dst);
#pragma unroll
        for (int i = 0; i < 4; ++i) q[i] = make_float4(u[4 * i], u[4 * i + 1], u[4 * i + 2], u[4 * i + 3]);
        reinterpret_cast<float2*>(dst)[8] = make_float2(u[16], u[17]);
    } else {
        double2* q = reinterpret_cast<double2*>(dst);
#pragma unroll
        for (int i = 0; i < 9; ++i) q[i] = make_double2(u[2 * i], u[2 * i + 1]);
    }
}

// CTA tile: NS 4D sites x Ls slices, one thread per 5D site.  Bit 0 of the
// variant picks the shape: 0 the default, 1 twice the sites (half for
// Ls = 12).  Bit 1 caps the registers at about 72 per thread (one more
// resident CTA of 128 threads than the compiler's own choice of 80, a few
// spilled values) and applies to FP32 arithmetic only.  The autotuner
// times the variants for the inner-solver kinds.
template <int LS, int VAR = 0> struct Tile {
    static constexpr int NS0 = (LS >= 16) ? 8 : (LS == 12 ? 16 : 128 / LS);
    static constexpr int NS = (VAR & 1) == 0 ? NS0 : (LS == 12 ? NS0 / 2 : NS0 * 2);
    static constexpr int NT = NS * LS;
};

template <typename S> constexpr int kTileVariants = sizeof(typename Traits<S>::R) == 4 ? 4 : 2;

// the register-capped variants ask for this many resident CTAs per SM
template <int LS, int VAR> struct MinBlocksCap {
    static constexpr int V = 65536 / (72 * Tile<LS, VAR>::NT);
};

// lanes per 5D site of a kernel (the FP64 hop kinds: two, one per upper spin),
// and its CTA: the FP64 hop kinds take half the sites of the tile (against one
// lane per site on the same half tile, when both were FP64 hops without the
// FP64 fallback: K at 4^4 Ls = 8 53 -> 37 us, FP64 CG iteration at 8^3x16
// Ls = 8 157 -> 133 us, K^dag at 24^3x64 Ls = 12 8.85 -> 6.94 ms; K at
// 16^3x32 Ls = 16 1.15 -> 1.20 ms lost).  The two applications with a column
// phase take a quarter at Ls = 12: CTAs of three warps leave room for five,
// with 128 registers, where those of six leave room for two (168) or three
// (96).  4 sites, 8 sites in three CTAs: K^dag 354, 363 us and H 342, 359 us at
// 12^3x24; K^dag 2.79, 2.84 ms at 24^4.  K itself, 4 sites or 8 in two CTAs:
// 2.61, 2.49 ms at 24^4.
template <typename S, int LS, int K, int VAR> struct HopTile {
    static constexpr int HV = sizeof(S) == 8 && KindTraits<K>::HOP ? 2 : 1;
    static constexpr bool QUARTER = HV == 2 && LS == 12 && (K == KIND_FULL_DAG || K == KIND_H);
    static constexpr int NS = Tile<LS, VAR>::NS / (QUARTER ? 4 : HV);
    static constexpr int NT = NS * LS * HV;
};

// sites per CTA of a tile variant of the inner kinds (for reports)
inline int tile_sites(int prec, int Ls, int var) {
    const bool alt = var & 1;
    if (prec == 0) return tile_sites(1, Ls, var) / 2;
    switch (Ls) {
        case 4: return alt ? Tile<4, 1>::NS : Tile<4, 0>::NS;
        case 8: return alt ? Tile<8, 1>::NS : Tile<8, 0>::NS;
        case 12: return alt ? Tile<12, 1>::NS : Tile<12, 0>::NS;
        case 16: return alt ? Tile<16, 1>::NS : Tile<16, 0>::NS;
        default: return 0;
    }
}

// raw link records (rows 0 and 1 in storage precision) are staged with
// cp.async, 16-byte pieces (8-byte for 16-bit storage)
template <typename S> struct LinkRaw {
    static constexpr int BYTES = 12 * (int)sizeof(S);
    // storage = compute precision: the record lands in rows 0-1 of its
    // staged link and row 2 is rebuilt in place; 16-bit storage needs a
    // separate raw buffer
    static constexpr bool SEP = sizeof(S) != sizeof(typename Traits<S>::R);
    static constexpr int PAD = SEP ? (BYTES + 15) / 16 * 16 : 0;
};

__device__ __forceinline__ void stage_cp16(void* dst, const void* src) {
    const unsigned sa = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(sa), "l"(src) : "memory");
}
__device__ __forceinline__ void stage_cp8(void* dst, const void* src) {
    const unsigned sa = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(sa), "l"(src) : "memory");
}
__device__ __forceinline__ void stage_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
__device__ __forceinline__ void stage_wait() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }

// one staged raw link record -> 12 reals of compute precision
template <typename S, typename R>
__device__ __forceinline__ void link_from_raw(const unsigned char* raw, R* u) {
    if constexpr (sizeof(S) == 8) {
        const double2* p = reinterpret_cast<const double2*>(raw);
#pragma unroll
        for (int c = 0; c < 6; ++c) {
            const double2 t = p[c];
            u[2 * c] = t.x;
            u[2 * c + 1] = t.y;
        }
    } else if constexpr (sizeof(S) == 4) {
        const float4* p = reinterpret_cast<const float4*>(raw);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const float4 t = p[c];
            u[4 * c] = t.x;
            u[4 * c + 1] = t.y;
            u[4 * c + 2] = t.z;
            u[4 * c + 3] = t.w;
        }
    } else {
        const uint2* p = reinterpret_cast<const uint2*>(raw);
#pragma unroll
        for (int c = 0; c < 3; ++c) unpack4(p[c], (const S*)nullptr, u + 4 * c);
    }
}

// lanes and the other lanes of their sites
__device__ __forceinline__ unsigned hop_sites(unsigned lanes) {
    return lanes | ((lanes & 0x55555555u) << 1) | ((lanes >> 1) & 0x55555555u);
}

// The reals of hop_fixed's sums that some term is not exactly zero in: bit i
// for up[i], bit 6 + i for lo[i] (as they are at the end).  A fixed-point real
// and an element of rows 0 and 1 of a staged link are zero only if the double
// is (fx_from); row 2 goes by its cofactors.  Sparse fields on links that keep
// them sparse (a point source in the free field) have many exact zeros.
static __device__ __forceinline__ unsigned hop_terms(const HopArgs* __restrict__ a, const int4* __restrict__ lk,
                                                  const unsigned* __restrict__ nb, int s, int sp, int Ls,
                                                  unsigned mask) {
    unsigned up = 0, lo = 0;
    auto swap = [](unsigned m) { return ((m & 0x15u) << 1) | ((m >> 1) & 0x15u); };
#pragma unroll 1
    for (int k = 0; k < 8; ++k) {
        const int mu = k >> 1, low = mu < 2 ? 3 - sp : 2 + sp;
        const bool back = k & 1, real = mu & 1;
        if (k == 4) lo = __shfl_xor_sync(mask, lo, 1);
        const longlong2* q = reinterpret_cast<const longlong2*>(a->in) +
                             (long)(nb[4 * back + mu] & 0x7fffffffu) * 12 * Ls + s;
        unsigned h[2] = {0, 0};  // real and imaginary parts of h, a bit a colour
        for (int b = 0; b < 3; ++b) {
            const longlong2 v = q[(3 * sp + b) * Ls], y = q[(3 * low + b) * Ls];
            h[0] |= (unsigned)((v.x | (real ? y.x : y.y)) != 0) << b;
            h[1] |= (unsigned)((v.y | (real ? y.y : y.x)) != 0) << b;
        }
        unsigned u[3][2] = {};  // rows of U, a bit a column
        const int4* W = lk + (4 * back + mu) * 9;
        for (int r = 0; r < 2; ++r)
            for (int c = 0; c < 3; ++c) {
                const int4 e = W[back ? 3 * c + r : 3 * r + c];
                u[r][0] |= (unsigned)((e.x | e.y) != 0) << c;
                u[r][1] |= (unsigned)((e.z | e.w) != 0) << c;
            }
        auto next = [](unsigned m, int n) { return ((m | m << 3) >> n) & 7u; };  // bit c takes bit c + n (mod 3)
        for (int i = 0; i < 2; ++i)
            for (int j = 0; j < 2; ++j)
                u[2][i ^ j] |= (next(u[0][i], 1) & next(u[1][j], 2)) | (next(u[0][i], 2) & next(u[1][j], 1));
        unsigned w = 0;  // W h in the order of up
        for (int c = 0; c < 3; ++c)
            for (int b = 0; b < 3; ++b)
                for (int i = 0; i < 2; ++i)
                    for (int j = 0; j < 2; ++j)
                        w |= ((back ? u[b][i] >> c : u[c][i] >> b) & (h[j] >> b) & 1u) << (2 * c + (i ^ j));
        up |= w;
        lo |= real ? w : swap(w);
    }
    return up | lo << 6;
}

// The hop sum of one 5D site in FP64 arithmetic by the two lanes of hop_fixed,
// from the doubles behind the hop input and the links as stored: the sites
// whose sums the integers cannot hold (fixed64.cuh).  small: the reals without
// a large term (bits as in hop_terms), or bit 31 where a neighbour has no
// integers; false, and nothing done, where the small ones are exact zeros.
// pre: the input takes D~ / b5 (z, mz as in chi).  mask: the lanes that call,
// both of a site.  Ls and fs are runtime values and one call serves both
// steps: one copy for all kernels, few values to keep across it (two calls: H
// at 24^3x64, Ls = 12 7.36 ms, one 7.20).  16^4, Ls = 16, all sites in FP64: K
// 3.2 to 3.9 ms (2.36 ms for a kernel of FP64 arithmetic alone); all with zeros
// that stay: 0.78 ms.
static __device__ __noinline__ bool hop_fp64(const HopArgs* __restrict__ a, const int4* __restrict__ lk,
                                             const unsigned* __restrict__ nb, long xcb, int s, int sp, int Ls, int fs,
                                             bool pre, double z, double mz, unsigned mask, unsigned small,
                                             double* __restrict__ out) {
    const bool raw = small >> 31;
    const unsigned held = __ballot_sync(mask, !raw);  // both lanes of a site alike
    if (!raw) small &= hop_terms(a, lk, nb, s, sp, Ls, held);
    mask = hop_sites(__ballot_sync(mask, small != 0));
    if (!(mask >> (threadIdx.x & 31) & 1)) return false;
    const bool canon = a->canon & 1;
    const int cs = canon ? 1 : Ls, ss = canon ? 12 : 1;  // strides of components and of slices
    double up[6], lo[6];
#pragma unroll
    for (int i = 0; i < 6; ++i) up[i] = lo[i] = 0.0;
#pragma unroll 1
    for (int k = 0; k < 8; ++k) {
        const int mu = k >> 1;
        const bool back = k & 1;
        const unsigned e = nb[4 * back + mu];
        const long n = (long)(e & 0x7fffffffu);
        if (k == 4) {  // the lower sums so far belong to the other lane
#pragma unroll
            for (int i = 0; i < 6; ++i) lo[i] = __shfl_xor_sync(mask, lo[i], 1);
        }
        const double2* p = reinterpret_cast<const double2*>(a->in_raw) +
                           (canon ? lex_site(a->g, n, 1 - a->out_par) : n) * 12 * Ls;
        auto load = [&](int spin, int b) {
            const double2* q = p + (3 * spin + b) * cs;
            double2 v = q[s * ss];
            if (pre) {
                const bool edge = spin < 2 ? s == 0 : s == Ls - 1;
                const double2 w = q[(spin < 2 ? (edge ? Ls - 1 : s - 1) : (edge ? 0 : s + 1)) * ss];
                const double f = edge ? -mz : z;
                v.x += f * w.x;
                v.y += f * w.y;
            }
            return v;
        };
        // h = psi_sp + f psi_low (mu = 1, 3) or psi_sp + i f psi_low
        const bool real = mu & 1;
        const double f = (back ? -fs : fs) * (mu == 0 || (mu != 3 && sp == 0) ? -1.0 : 1.0);
        double2 h[3];
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            const double2 v = load(sp, b), y = load(mu < 2 ? 3 - sp : 2 + sp, b);
            h[b] = make_double2(fma(f, real ? y.x : -y.y, v.x), fma(f, real ? y.y : y.x, v.y));
        }
        const double* rec = reinterpret_cast<const double*>(back ? a->lk_in : a->lk_out) +
                            ((back ? n : xcb) * 4 + mu) * 12;
        double u[18];
#pragma unroll
        for (int i = 0; i < 12; ++i) u[i] = rec[i];
        // row 2 = conj(row 0 x row 1): lane 0 makes its real parts, lane 1 the imaginary ones
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            const double* a1 = u + 2 * ((q + 1) % 3);
            const double* a2 = u + 2 * ((q + 2) % 3);
            const double *b1 = a1 + 6, *b2 = a2 + 6;
            const double p1 = sp ? -b2[1] : b2[0], p2 = sp ? -b2[0] : -b2[1];
            const double q1 = sp ? -b1[1] : b1[0], q2 = sp ? -b1[0] : -b1[1];
            const double mine = (a1[0] * p1 + a1[1] * p2) - (a2[0] * q1 + a2[1] * q2);
            const double other = __shfl_xor_sync(mask, mine, 1);
            u[12 + 2 * q] = sp ? other : mine;
            u[13 + 2 * q] = sp ? mine : other;
        }
        const bool neg = e >> 31;  // the boundary sign
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            if (neg) h[b] = make_double2(-h[b].x, -h[b].y);
        }
        double2 w[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) w[c] = make_double2(0.0, 0.0);
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            if (h[b].x == 0.0 && h[b].y == 0.0) continue;  // the links are finite
#pragma unroll
            for (int c = 0; c < 3; ++c) {  // U_cb, or conj(U_bc)
                const int i = 6 * c + 2 * b, j = 6 * b + 2 * c;
                const double x = back ? u[j] : u[i], y = back ? -u[j + 1] : u[i + 1];
                w[c].x = fma(x, h[b].x, fma(-y, h[b].y, w[c].x));
                w[c].y = fma(x, h[b].y, fma(y, h[b].x, w[c].y));
            }
        }
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            up[2 * c] += w[c].x;
            up[2 * c + 1] += w[c].y;
            lo[2 * c] = fma(f, real ? w[c].x : w[c].y, lo[2 * c]);
            lo[2 * c + 1] = fma(f, real ? w[c].y : -w[c].x, lo[2 * c + 1]);
        }
    }
#pragma unroll
    for (int i = 0; i < 6; ++i) {
        out[i] = up[i];
        out[6 + i] = lo[i];
    }
    return true;
}

// The hop sum of one 5D site in fixed point (fixed64.cuh) by two lanes: lane
// sp forms the projected colour vector h = psi_sp + sigma B psi_low, its
// product w, and adds w to spin sp and sigma B^dag w to a lower spin, 3 - sp
// for mu = 0, 1 and 2 + sp for mu = 2, 3.  After mu = 1 the lanes swap their
// lower sums, so each ends with spins sp and 2 + sp.  sigma is the projector's
// sign times the lane's sign in B (mu = 1: -, +; mu = 2: +, -); a lane takes
// the direction with sigma = +1 first, so that the sign is the same for all.
// Per lane: half the loads, products and sums of one lane for the site.  lk: the
// site's 8 staged links (backward ones daggered), nb its neighbour indices,
// mask: the lanes that call.  Two mu at a time: four copies of the products fit
// the instruction cache, eight do not.  The units known beforehand and the
// test for small terms cost 2 to 7% of the kernel (H at 24^3x64, Ls = 12 6.73 ->
// 7.20 ms, K at 16^4, Ls = 16 598 -> 608 us, an FP64 CG iteration 1340 -> 1364).
template <int LS, bool DAG, bool PRE>
__device__ __forceinline__ void hop_fixed(const HopArgs& a, const SCoef<double>& cf, const int4* __restrict__ lk,
                                          const unsigned* __restrict__ nb, long xcb, int s, int sp, unsigned mask,
                                          double* out) {
    const longlong2* base = reinterpret_cast<const longlong2*>(a.in) + s;
    const int* ex = reinterpret_cast<const int*>(a.in_nrm) + s;
    i64 up[6], lo[6];
#pragma unroll
    for (int i = 0; i < 6; ++i) up[i] = lo[i] = 0;
    // E, the exponent field of the units of the sums, is the neighbours'
    // largest; shl, shh: a byte for each direction, how far its own lies below
    int E = 0;
    unsigned shl = 0, shh = 0;
    {
        int e[8];
#pragma unroll
        for (int l = 0; l < 8; ++l) {
            e[l] = ex[(long)(nb[l] & 0x7fffffffu) * LS];
            E = max(E, e[l]);
        }
#pragma unroll
        for (int l = 0; l < 4; ++l) {
            shl |= (unsigned)min(E - e[l], 63) << (8 * l);
            shh |= (unsigned)min(E - e[4 + l], 63) << (8 * l);
        }
    }
    // a bit for each real of the upper and of the lower sums that some term of
    // size 2^-kFxSmall of the unit's 2^56 or more has gone into
    unsigned upm = 0, lom = 0;
    // B is -i times real for mu = 0, 2 and real for mu = 1, 3
    auto step = [&](auto real_c, auto plus_c, int l, int low) {
        constexpr bool REAL = decltype(real_c)::value, PLUS = decltype(plus_c)::value;
        const long n = (long)(nb[l] & 0x7fffffffu);
        const longlong2* q = base + n * (12 * LS);
        const longlong2* qu = q + 3 * sp * LS;
        const longlong2* ql = q + low * LS;
        i64 h[6], w[6];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const longlong2 t = qu[c * LS], b = ql[c * LS];
            if constexpr (REAL) {
                h[2 * c] = PLUS ? t.x + b.x : t.x - b.x;
                h[2 * c + 1] = PLUS ? t.y + b.y : t.y - b.y;
            } else {
                h[2 * c] = PLUS ? t.x + b.y : t.x - b.y;
                h[2 * c + 1] = PLUS ? t.y - b.x : t.y + b.x;
            }
        }
        const int sh = __byte_perm(shl, shh, l) & 63;
        const i64 half = (i64)((1ull << sh) >> 1);
#pragma unroll
        for (int i = 0; i < 6; ++i) h[i] = (h[i] + half) >> sh;
        fx_mul(lk + l * 9, h, w);
        unsigned big = 0;
#pragma unroll
        for (int i = 0; i < 6; ++i) {
            constexpr unsigned T = 1u << (kFxFrac - 32 - kFxSmall);
            if ((unsigned)((int)(w[i] >> 32)) + T >= 2 * T) big |= 1u << i;
        }
        upm |= big;
        lom |= REAL ? big : ((big & 0x15u) << 1) | ((big >> 1) & 0x15u);
#pragma unroll
        for (int i = 0; i < 6; i += 2) {
            up[i] += w[i];
            up[i + 1] += w[i + 1];
            if constexpr (REAL) {
                lo[i] = PLUS ? lo[i] + w[i] : lo[i] - w[i];
                lo[i + 1] = PLUS ? lo[i + 1] + w[i + 1] : lo[i + 1] - w[i + 1];
            } else {
                lo[i] = PLUS ? lo[i] - w[i + 1] : lo[i] + w[i + 1];
                lo[i + 1] = PLUS ? lo[i + 1] + w[i] : lo[i + 1] - w[i];
            }
        }
    };
    // the projector is 1 + gamma forward for D^dag and backward for D
    constexpr int BACK = DAG ? 0 : 4;
    typedef std::integral_constant<bool, true> T;
    typedef std::integral_constant<bool, false> F;
#pragma unroll 1
    for (int half = 0; half < 2; ++half) {  // mu = 0, 1, then 2, 3
        const int fi = half ? 4 * sp : 0, fr = half ? 0 : 4 * (1 - sp);
        const int low = 6 + 3 * (half ? sp : 1 - sp), l = 2 * half;
        step(F{}, T{}, l + (fi ^ BACK), low);
        step(F{}, F{}, l + (fi ^ BACK ^ 4), low);
        step(T{}, T{}, l + 1 + (fr ^ BACK), low);
        step(T{}, F{}, l + 1 + (fr ^ BACK ^ 4), low);
        if (half == 0) {  // both lanes have the same unit
#pragma unroll
            for (int i = 0; i < 6; ++i) lo[i] = __shfl_xor_sync(mask, lo[i], 1);
            lom = __shfl_xor_sync(mask, lom, 1);
        }
    }
#pragma unroll
    for (int i = 0; i < 6; ++i) {
        out[i] = fx_to(up[i], E);
        out[6 + i] = fx_to(lo[i], E);
    }
    // sites for FP64 arithmetic (E = 0: every neighbour is zero)
    const unsigned small = E == kFxRaw ? 1u << 31 : E > 0 ? ~(upm | lom << 6) & 0xfffu : 0u;
    const unsigned slow = hop_sites(__ballot_sync(mask, small != 0));
    if (slow >> (threadIdx.x & 31) & 1) {
        double r[12];
        if (hop_fp64(&a, lk, nb, xcb, s, sp, LS, DAG ? 1 : -1, PRE, cf.zb, cf.mzb, slow, small, r)) {
#pragma unroll
            for (int i = 0; i < 12; ++i) out[i] = r[i];
        }
    }
}

// Persistent CTAs: a CTA walks the site blocks blockIdx.x, +gridDim.x, ...
// While it works on one block, the links and neighbour indices of its next
// block are already on their way (cp.async into a second staging buffer),
// so the link latency is off the critical path, and the norm reduction runs
// once per CTA instead of once per block.
template <typename S, int LS, int KIND, int VAR>
__device__ __forceinline__ void hop_body(const HopArgs& a, const SCoef<typename Traits<S>::R>& cf) {
    typedef typename Traits<S>::R R;
    typedef KindTraits<KIND> KT;
    constexpr int HV = HopTile<S, LS, KIND, VAR>::HV;
    constexpr int NS = HopTile<S, LS, KIND, VAR>::NS;
    constexpr int NT = HopTile<S, LS, KIND, VAR>::NT;
    constexpr int NR = 24 / HV, HF = 12 / HV;  // reals of a lane: HF of each chirality
    constexpr int NCOL = sizeof(R) == 8 ? 24 : 12;  // columns of a site (ColVal)
    constexpr int ST = ShStride<R>::V;
    constexpr int SS = SiteStride<R, LS>::V;
    constexpr int LK = LinkStride<R>::V;
    constexpr int NL = NS * 8;  // staged links (and neighbour indices) per block
    constexpr int RAWB = LinkRaw<S>::PAD;
    constexpr bool FX = sizeof(S) == 8;  // the hop in fixed point (fixed64.cuh)
    constexpr bool CANON = FX && KT::APPLY;

    // issued now, used after the first links are staged; a launch of several
    // blocks per CTA, whose first stage is a small part, leaves at once
    const int dn = a.done ? *reinterpret_cast<const volatile int*>(a.done) : 0;
    auto leave = [&]() {
        if (a.stop && blockIdx.x == 0 && threadIdx.x == 0) *a.stop = 1;
    };
    if ((long)gridDim.x * NS < a.g.Vh && dn) return leave();

    extern __shared__ __align__(16) unsigned char smem_raw[];
    constexpr bool SHF = ShflTail<KIND, LS>::ON;
    constexpr bool COLS = ShflTail<KIND, LS>::COLS;  // column phase and its tile buffers
    R* sh = reinterpret_cast<R*>(smem_raw);          // [NS][SS] hop result
    R* sy = sh + (COLS ? NS * SS : 0);                // [NS][SS] local input
    R* smat = sy + ((KT::HASY && COLS && !KT::YCOL) ? NS * SS : 0);  // [2][LS][LS] dense kinds' s-matrices
    R* sl = smat + (KT::DENSE ? 2 * LS * LS : 0);       // [2][NL][LK] links, row 2 rebuilt
    unsigned char* sraw = reinterpret_cast<unsigned char*>(sl + (KT::HOP ? 2 * NL * LK : 0));  // [2][NL][RAWB]
    unsigned* snb = reinterpret_cast<unsigned*>(sraw + (KT::HOP ? 2 * NL * RAWB : 0));        // [2][NL]

    const Geom& g = a.g;
    const int tid = threadIdx.x;
    const int il = tid / (LS * HV);
    const int s = (tid - il * LS * HV) / HV;
    const int sp = tid % HV;                                    // the lane's upper spin (HV = 2)
    const int rp = il * SS + s * ST + sp * HF;                  // row of the P+ half
    const int rm = il * SS + (LS - 1 - s) * ST + 12 + sp * HF;  // row of the P- half
    const long nblk = ((long)g.Vh + NS - 1) / NS;
    // ---------------- phase 0: links and neighbours, once per 4D site ---
    // The 8 links of each site (4 forward from this parity, 4 backward from
    // the neighbours) and the 8 neighbour indices (bit 31: the hop carries a
    // factor -1, from an antiperiodic or a G-parity boundary) for all Ls
    // slices of the site.  Issue: indices and
    // cp.async of the raw records; finish: the third row rebuilt.
    auto stage_issue = [&](long blk, int b) {
        for (int j = tid; j < NL; j += NT) {
            const int jl = j >> 3, d = j & 7, mu = d & 3;
            const long jcb = blk * NS + jl;
            if (jcb < g.Vh) {
                int rem = (int)jcb;
                const int xh = rem % g.Xh; rem /= g.Xh;
                const int y = rem % g.Y; rem /= g.Y;
                const int z = rem % g.Z;
                const int tf = rem / g.Z;  // t + f Tp for flavour f (G-parity), else t
                const int x = 2 * xh + ((a.out_par + y + z + tf) & 1);
                const int f = tf >= g.Tp ? 1 : 0;
                // step in direction mu (forward for d < 4), periodic wrap
                const int c = mu == 0 ? x : mu == 1 ? y : mu == 2 ? z : tf - f * g.Tp;
                const int e = mu == 0 ? g.X : mu == 1 ? g.Y : mu == 2 ? g.Z : g.Tp;
                const bool cross = (d < 4) ? (c + 1 == e) : (c == 0);
                const int n = (d < 4) ? (cross ? 0 : c + 1) : (cross ? e - 1 : c - 1);
                long ncb = ((((long)(mu == 3 ? n + f * g.Tp : tf) * g.Z + (mu == 2 ? n : z)) * g.Y +
                             (mu == 1 ? n : y)) * g.X + (mu == 0 ? n : x)) >> 1;
                bool neg = cross && ((g.apmask >> mu) & 1);
                if (cross && ((g.gpmask >> mu) & 1)) {
                    // G-parity boundary: psi_1(x + L) = psi_2(x), psi_2(x + L) = -psi_1(x);
                    // the other flavour is half the stacked lattice away
                    ncb += f ? -(long)(g.Vh / 2) : (long)(g.Vh / 2);
                    neg = neg != ((d < 4) ? f == 1 : f == 0);
                }
                const unsigned edge = neg ? 0x80000000u : 0u;
                snb[b * NL + j] = (unsigned)ncb | edge;
                const long site = (d < 4) ? jcb : ncb;
                const unsigned char* src = reinterpret_cast<const unsigned char*>(d < 4 ? a.lk_out : a.lk_in) +
                                           (site * 4 + mu) * LinkRaw<S>::BYTES;
                unsigned char* dst = LinkRaw<S>::SEP ? sraw + (b * NL + j) * RAWB
                                                     : reinterpret_cast<unsigned char*>(sl + (b * NL + j) * LK);
                if constexpr (sizeof(S) >= 4) {
#pragma unroll
                    for (int c = 0; c < LinkRaw<S>::BYTES / 16; ++c) stage_cp16(dst + 16 * c, src + 16 * c);
                } else {
#pragma unroll
                    for (int c = 0; c < 3; ++c) stage_cp8(dst + 8 * c, src + 8 * c);
                }
            }
        }
        stage_commit();
    };
    auto stage_finish = [&](long blk, int b) {
        stage_wait();  // this thread's own copies
        for (int j = tid; j < NL; j += NT) {
            if (blk * NS + (j >> 3) < g.Vh) {
                R u[18];
                R* dl = sl + (b * NL + j) * LK;
                if constexpr (LinkRaw<S>::SEP) link_from_raw<S, R>(sraw + (b * NL + j) * RAWB, u);
                else link_from_raw<S, R>(reinterpret_cast<const unsigned char*>(dl), u);
                if constexpr (FX) {
                    fx_stage_link(u, (g.gpmask | g.apmask) && (snb[b * NL + j] >> 31), (j & 7) >= 4,
                                  reinterpret_cast<int4*>(dl));
                    continue;
                }
                rebuild_row2(u);
                // the factor -1 of an antiperiodic or G-parity boundary hop
                // rides on the staged link; the branch is uniform over the grid
                if ((g.gpmask | g.apmask) && (snb[b * NL + j] >> 31)) {
#pragma unroll
                    for (int i = 0; i < 18; ++i) u[i] = -u[i];
                }
                st_link(dl, u);
            }
        }
    };

    long blk = blockIdx.x;
    if constexpr (KT::DENSE) {  // published by the barrier after the first links
        const R* gm = reinterpret_cast<const R*>(a.dense);
        for (int i = tid; i < 2 * LS * LS; i += NT) smat[i] = gm[i];
    }
    if constexpr (KT::HOP) {
        if (blk < nblk) {
            stage_issue(blk, 0);
            stage_finish(blk, 0);
        }
        __syncthreads();
    }
    if (dn) return leave();

    R nn = (R)0;
    for (int it = 0; blk < nblk; ++it, blk += gridDim.x) {
        const int cur = it & 1;
        const long nxt = blk + gridDim.x;
        if constexpr (KT::HOP) {
            if (nxt < nblk) stage_issue(nxt, cur ^ 1);
        }
        const R* slc = sl + cur * NL * LK;
        const unsigned* snc = snb + cur * NL;
        const long xcb = blk * NS + il;
        const bool valid = xcb < g.Vh;
        const unsigned mask = HV == 2 ? __ballot_sync(0xffffffffu, valid) : 0u;

        // the site-local input, and the canonical site where the fields are the caller's
        long lex = 0;
        if constexpr (CANON) {
            if (a.canon && valid) lex = lex_site(g, xcb, a.out_par);
        }
        auto y_half = [&](int sl, int hi, R* q) {
            if constexpr (CANON) {
                if (a.canon) {
                    const double2* p = reinterpret_cast<const double2*>(a.y) + (lex * LS + sl) * 12 + 6 * hi + 3 * sp;
#pragma unroll
                    for (int c = 0; c < HF / 2; ++c) {
                        const double2 t = p[c];
                        q[2 * c] = t.x;
                        q[2 * c + 1] = t.y;
                    }
                    return;
                }
            }
            load_half_part<S, R, HV>(a.y, a.y_nrm, xcb, sl, LS, hi, sp, q);
        };
        auto y_load = [&](R* v) {
            if constexpr (CANON) {
                if (a.canon) {
                    y_half(s, 0, v);
                    y_half(s, 1, v + HF);
                    return;
                }
            }
            if constexpr (HV == 2) {
                load_half_part<S, R, HV>(a.y, a.y_nrm, xcb, s, LS, 0, sp, v);
                load_half_part<S, R, HV>(a.y, a.y_nrm, xcb, s, LS, 1, sp, v + HF);
            } else {
                load_sp<S, R>(a.y, a.y_nrm, xcb, s, LS, v);
            }
        };

        if constexpr (KT::YCOL) {
            if (valid) {
                R v[NR];
                y_load(v);
                st_half<HF>(sh + rp, v);
                st_half<HF>(sh + rm, v + HF);
            }
            __syncthreads();
            for (int col = tid; col < NS * NCOL; col += NT) {
                const int ci = col / NCOL;
                const int cc = (col - ci * NCOL) * (24 / NCOL);  // place among the 24 reals of a row
                const bool shv = cf.has_shift && ((cc >= 12 ? 1 : 0) == cf.cs);
                column_program<R, LS, KIND, ST>(sh + ci * SS + cc, (const R*)nullptr, cf, shv, (R)1, (const R*)nullptr);
            }
        }

        // ---------------- phase 1: hop and staging ----------------------
        R o[NR];    // the output spinor of this thread's 5D site
        R acc[NR];  // its hop result (zero for padding sites)
#pragma unroll
        for (int i = 0; i < NR; ++i) acc[i] = (R)0;
        if (valid) {
            if constexpr (KT::HOP) {
                constexpr int FS = KT::DAG ? +1 : -1;  // forward projector 1 + FS gamma
                if constexpr (FX) {
                    hop_fixed<LS, KT::DAG, KT::PRE>(a, cf, reinterpret_cast<const int4*>(slc + il * 8 * LK),
                                                    snc + il * 8, xcb, s, sp, mask, acc);
                } else
                // hop k = 2 mu + dir (dir 0 forward, 1 backward)
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    const int mu = k >> 1, dir = k & 1;
                    const long ncb = (long)(snc[il * 8 + dir * 4 + mu] & 0x7fffffffu);
                    R p[24];
                    load_sp<S, R>(a.in, a.in_nrm, ncb, s, LS, p);
                    if constexpr (KT::PRE) {
                        // chi = psi + (c5/b5) L psi (the b5 factor is applied in phase 2)
                        R q[12];
                        const int sm = (s == 0) ? LS - 1 : s - 1;
                        const R fu = (s == 0) ? -cf.mzb : cf.zb;
                        load_half<S, R>(a.in, a.in_nrm, ncb, sm, LS, 0, q);
#pragma unroll
                        for (int i = 0; i < 12; ++i) p[i] += fu * q[i];
                        const int sp = (s == LS - 1) ? 0 : s + 1;
                        const R fd = (s == LS - 1) ? -cf.mzb : cf.zb;
                        load_half<S, R>(a.in, a.in_nrm, ncb, sp, LS, 1, q);
#pragma unroll
                        for (int i = 0; i < 12; ++i) p[12 + i] += fd * q[i];
                    }
                    R u[18];
                    ld_link(slc + (il * 8 + dir * 4 + mu) * LK, u);
                    // every boundary sign rides on the staged link
                    if (dir == 0) {
                        if (mu == 0) hop_dir<R, 0, FS, false>(acc, p, u);
                        if (mu == 1) hop_dir<R, 1, FS, false>(acc, p, u);
                        if (mu == 2) hop_dir<R, 2, FS, false>(acc, p, u);
                        if (mu == 3) hop_dir<R, 3, FS, false>(acc, p, u);
                    } else {
                        if (mu == 0) hop_dir<R, 0, -FS, true>(acc, p, u);
                        if (mu == 1) hop_dir<R, 1, -FS, true>(acc, p, u);
                        if (mu == 2) hop_dir<R, 2, -FS, true>(acc, p, u);
                        if (mu == 3) hop_dir<R, 3, -FS, true>(acc, p, u);
                    }
                }
                if constexpr (KT::PTW) {
                    // out = [M] y + f h, finished in registers
                    const R f = ((KIND == KIND_FULL) ? (R)-0.5 : (R)0.5) * (KT::PRE ? cf.b5 : (R)1);
                    R v[NR];
                    y_load(v);
                    if constexpr (KIND != KIND_SRC) site_M<R, LS, HF>(y_half, s, cf, v);
#pragma unroll
                    for (int i = 0; i < NR; ++i) o[i] = v[i] + f * acc[i];
                } else if constexpr (COLS && !KT::YCOL) {
                    st_half<HF>(sh + rp, acc);
                    st_half<HF>(sh + rm, acc + HF);
                }
            }
            if constexpr (KT::HASY && COLS && !KT::YCOL) {
                R v[NR];
                y_load(v);
                st_half<HF>(sy + rp, v);
                st_half<HF>(sy + rm, v + HF);
            }
        }
        if constexpr (SHF) {
            // out = M^T y + f D~^T h with the slice neighbours from the site's lanes
            R v[NR];
            if (valid) {
                y_load(v);
            } else {
#pragma unroll
                for (int i = 0; i < NR; ++i) v[i] = (R)0;
            }
            const R f = (KIND == KIND_FULL_DAG) ? (R)-0.5 : (R)0.5;
            site_MT_dtT<R, LS, HV>(s, sp, cf, v, acc, f, o);
        }

        // ---------------- phase 2: fifth-dimension program --------------
        if constexpr (KT::YCOL) {
            __syncthreads();
        } else if constexpr (COLS) {
            __syncthreads();
            const R hb = KT::PRE ? cf.b5 : (R)1;  // the b5 of the on-the-fly D~
            for (int col = tid; col < NS * NCOL; col += NT) {
                const int ci = col / NCOL;
                const int cc = (col - ci * NCOL) * (24 / NCOL);  // place among the 24 reals of a row
                const bool shv = cf.has_shift && ((cc >= 12 ? 1 : 0) == cf.cs);
                column_program<R, LS, KIND, ST>(sh + ci * SS + cc, sy + ci * SS + cc, cf, shv, hb,
                                                smat + (cc >= 12 ? LS * LS : 0));
            }
            __syncthreads();
        }

        // ---------------- phase 3: store ----------------------------------
        if (valid) {
            if constexpr (COLS) {
                ld_half<HF>(sh + rp, o);
                ld_half<HF>(sh + rm, o + HF);
            }
            if constexpr (KT::YCOL) {
#pragma unroll
                for (int i = 0; i < NR; ++i)
                    o[i] = KIND == KIND_H ? cf.kTi * o[i] - (R)0.5 * acc[i] : o[i] + cf.fR * acc[i];
            }
            void* out = a.out;
            if constexpr (FX && KT::FXOUT) {
                if constexpr (HV == 2) fx_store_part(out, a.out_nrm, xcb, s, LS, sp, o, mask);
                else fx_store(out, a.out_nrm, xcb, s, LS, o);
                out = a.out_raw;
            }
            if (CANON && a.canon) {
                const bool g5 = a.canon & 2;
                double2* p = reinterpret_cast<double2*>(a.out) + (lex * LS + (g5 ? LS - 1 - s : s)) * 12 + 3 * sp;
                const double f = g5 ? -1.0 : 1.0;
#pragma unroll
                for (int c = 0; c < HF / 2; ++c) {
                    p[c] = make_double2(o[2 * c], o[2 * c + 1]);
                    p[6 + c] = make_double2(f * o[HF + 2 * c], f * o[HF + 2 * c + 1]);
                }
            } else if constexpr (HV == 2) {
                double2* p = reinterpret_cast<double2*>(out) + (xcb * 12 + 3 * sp) * LS + s;
#pragma unroll
                for (int c = 0; c < HF / 2; ++c) {
                    p[c * LS] = make_double2(o[2 * c], o[2 * c + 1]);
                    p[(6 + c) * LS] = make_double2(o[HF + 2 * c], o[HF + 2 * c + 1]);
                }
            } else {
                store_sp<S, R>(out, a.out_nrm, xcb, s, LS, o);
            }
            if (a.rd.fin != FIN_NONE) {
#pragma unroll
                for (int i = 0; i < NR; ++i) nn += o[i] * o[i];
            }
        }

        if constexpr (KT::HOP) {
            if (nxt < nblk) stage_finish(nxt, cur ^ 1);
        }
        __syncthreads();  // next block's links in place; this block's tiles free
    }
    if (a.rd.fin != FIN_NONE) block_reduce_finalize<NT>(nn, a.rd);
}

// Threads per SM that the FP64 hop kinds leave registers for (128 a thread).
// 512 against 640 threads: K at 16^4, Ls = 16 587 against 616 us, FP64 CG
// iteration 1357 against 1377 us, at 4^4, Ls = 8 76 against 80 us, at 12^3x24,
// Ls = 12 689 against 716 us; 768 threads lost everywhere.
constexpr int kFp64Threads = 512;

// the kernel with the compiler's own register choice (variants 0, 1) ...
template <typename S, int LS, int KIND, int VAR = 0>
__global__ void __launch_bounds__(HopTile<S, LS, KIND, VAR>::NT,
                                  HopTile<S, LS, KIND, VAR>::HV == 2 ? kFp64Threads / HopTile<S, LS, KIND, VAR>::NT : 1)
    hop_kernel(const __grid_constant__ HopArgs a, const SCoef<typename Traits<S>::R> cf) {
    hop_body<S, LS, KIND, VAR>(a, cf);
}

// ... an application's two parities in one grid (blockIdx.y) ...
struct HopPair {
    HopArgs a[2];
};
template <typename S, int LS, int KIND>
__global__ void __launch_bounds__(HopTile<S, LS, KIND, 0>::NT, kFp64Threads / HopTile<S, LS, KIND, 0>::NT)
    hop_kernel_pair(const __grid_constant__ HopPair p, const SCoef<typename Traits<S>::R> cf) {
    hop_body<S, LS, KIND, 0>(p.a[blockIdx.y], cf);
}

// ... and with capped registers (variants 2, 3; FP32 arithmetic)
template <typename S, int LS, int KIND, int VAR>
__global__ void __launch_bounds__(Tile<LS, VAR>::NT, MinBlocksCap<LS, VAR>::V)
    hop_kernel_rc(const __grid_constant__ HopArgs a, const SCoef<typename Traits<S>::R> cf) {
    hop_body<S, LS, KIND, VAR>(a, cf);
}

template <typename S, int LS, int K, int VAR = 0>
constexpr size_t hop_smem_bytes() {
    typedef typename Traits<S>::R R;
    constexpr size_t bufs = ShflTail<K, LS>::COLS ? (1 + (KindTraits<K>::HASY && !KindTraits<K>::YCOL ? 1 : 0)) : 0;
    constexpr size_t NS = HopTile<S, LS, K, VAR>::NS, NL = NS * 8;
    return bufs * NS * SiteStride<R, LS>::V * sizeof(R) +
           (KindTraits<K>::DENSE ? 2 * (size_t)LS * LS * sizeof(R) : 0) +
           (KindTraits<K>::HOP ? 2 * NL * (LinkStride<R>::V * sizeof(R) + LinkRaw<S>::PAD + sizeof(unsigned)) : 0);
}

}  // namespace eofa
