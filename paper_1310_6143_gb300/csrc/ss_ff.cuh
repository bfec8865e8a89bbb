// The thermal Gaussians of the FP32-mixed form: the Box-Muller transform of ss_math.cuh
// evaluated in double-float arithmetic (a value held as the unevaluated sum hi + lo of two
// floats, combined with error-free transformations: Dekker's product via FMA, Knuth's
// TwoSum and the fast two-sum for ordered operands), with a certified rounding to FP32.
//
// The FP32-mixed form stores the thermal field in FP32, so what its kernels need of the FP64
// transform is that transform's result rounded to FP32.  The double-float evaluation gets
// each Gaussian to within about 2^-44.5 (relative) of the exact value, on the FP32 pipes,
// and rounds it to FP32.  That rounding is accepted only when the double-float value lies
// further from the nearest rounding boundary (the midpoint between two floats) than an
// error bound that covers both the double-float evaluation and the FP64 transform
// (2^-41 |g| + 2^-43 R, R the Box-Muller radius; over 20 times the largest error seen in
// tests, and over 10 times the sum of the largest errors of each part over all 2^32
// inputs).  Both then round to the same float.  Otherwise (about four values in 10^5) the
// caller evaluates the FP64 transform and rounds its result.  Either way
// the float is exactly the FP64 transform's result rounded to nearest: the thermal field
// is bit for bit the same as with the FP64 transform, at a fraction of its cost on GB300,
// whose FP64 pipe issues two instructions per cycle per SM against 128 for FP32.
//
// Pieces (notation of ss_math.cuh: u = (w + 1/2) 2^-32 = m 2^-33, m = 2w + 1):
//   * -2 ln u: u = 2^-n f, f in [0.75, 1.5), nearest centre c = J/2048; f - c is an exact
//     multiple of 2^-33 (an integer below 2^23 times a power of two), r = (f - c)(1/c) with
//     1/c a double-float table entry; -2 ln(1 + r) = -2r + r^2 - r^3 (2/3 - r/2 + 2r^2/5)
//     (|r| < 3.3e-4, the r^3 tail in single precision); then + (-2 ln c) + 2 n ln 2, both
//     double-float table entries, added smallest first with the fast two-sum (each sum's
//     larger operand is known).
//   * sqrt(L): s0 = L rsqrt(L) in single precision, then two Newton corrections
//     c_k = (L - (s0 + c_1 + ..)^2) / (2 s0) whose residuals are formed exactly (Dekker's
//     product, FMAs).
//   * sin/cos of 2 pi u: the nearest of 4096 table angles a (one octant tabulated in
//     double-float, the rest by the exact symmetries of ss_math.cuh) and the remainder
//     d = 2 pi rho / 2^33 (|d| <= pi/4096) as a double-float product; sin(a + d) =
//     sin a + sin a (cos d - 1) + cos a sin d and its cosine counterpart, with
//     cos d - 1 = -d^2/2 + d^4/24 and sin d = d - d^3/6 (dropped terms below 1e-17).
//   * g = R cos, R sin: the double-float product, rounded to float with the check above.
#pragma once

#include <stdint.h>

#include "ss_math.cuh"

namespace ss {

// Shared-memory copy of the double-float tables (build_ff_tables):
//   lg[t]   = (1/c hi, 1/c lo, -2 ln c hi, -2 ln c lo), c = (kLogFirst + t) / kLogScale;
//   trig[m] = (sin hi, cos hi, sin lo, cos lo) of pi m / 2048, m = 0..512;
//   ln2[n]  = 2 n ln 2 (hi, lo), n = 0..33.
struct FFTables {
    float4 lg[kLogTab];
    float4 trig[kTrigTab];
    float2 ln2[kLn2Tab];
};

__device__ __forceinline__ void stage_ff_tables(const float4 *src, FFTables &t) {
    float4 *dst = reinterpret_cast<float4 *>(&t);
    for (int i = threadIdx.x; i < kLogTab + kTrigTab; i += blockDim.x) dst[i] = src[i];
    const float2 *s2 = reinterpret_cast<const float2 *>(src + kLogTab + kTrigTab);
    for (int i = threadIdx.x; i < kLn2Tab; i += blockDim.x) t.ln2[i] = s2[i];
}

struct FF {
    float hi, lo;
};

// a b = p + e exactly (Dekker's product through the FMA).
__device__ __forceinline__ FF ff_two_prod(float a, float b) {
    const float p = __fmul_rn(a, b);
    return FF{p, fmaf(a, b, -p)};
}

// a + b = s + e exactly (Knuth's TwoSum; no ordering of the operands needed).
__device__ __forceinline__ FF ff_two_sum(float a, float b) {
    const float s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    return FF{s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb))};
}

// a + b = s + e exactly when |a| >= |b| or a = 0 (the fast two-sum).
__device__ __forceinline__ FF ff_fast_two_sum(float a, float b) {
    const float s = __fadd_rn(a, b);
    return FF{s, __fsub_rn(b, __fsub_rn(s, a))};
}

// Two floats (two double-floats) side by side: one instruction of the packed FP32 forms
// (fma/add/mul.rn.f32x2) does both halves, each rounded as its scalar form is.  A Gaussian
// triple evaluates each of its functions twice -- two logarithms and square roots, two angles,
// the sine and cosine of the first -- so its two halves share every instruction but the integer
// ones and the table look-ups: 344 instructions a draw against 433 scalar ones (1024 x 1024 x 16
// film, 16 Heun steps: 10.47 -> 10.14 ms).
struct FFP {
    float2 hi, lo;
};
__device__ __forceinline__ float2 p2(float v) { return make_float2(v, v); }
__device__ __forceinline__ float2 p_neg(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ float2 p_mul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 p_add(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 p_fma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
// a - b: b (-1) is exact, so the fma rounds the difference once
__device__ __forceinline__ float2 p_sub(float2 a, float2 b) { return __ffma2_rn(b, p2(-1.0f), a); }

__device__ __forceinline__ FFP p_two_sum(float2 a, float2 b) {
    const float2 s = p_add(a, b);
    const float2 bb = p_sub(s, a);
    return FFP{s, p_add(p_sub(a, p_sub(s, bb)), p_sub(b, bb))};
}
__device__ __forceinline__ FFP p_fast_two_sum(float2 a, float2 b) {
    const float2 s = p_add(a, b);
    return FFP{s, p_sub(b, p_sub(s, a))};
}
__device__ __forceinline__ FFP p_add_ordered(FFP a, FFP b) {
    const FFP s = p_fast_two_sum(a.hi, b.hi);
    return p_fast_two_sum(s.hi, p_add(s.lo, p_add(a.lo, b.lo)));
}

// The integer part of -2 ln((w + 1/2) 2^-32): u = 2^-n f', f' in [0.75, 1.5), nearest centre
// c = J / 2048, dk = f' - c (exact).
__device__ __forceinline__ float ff_log_split(uint32_t w, uint32_t &J, int &n) {
    const int lz = __clz(w);
    // m = 2w + 1 with its leading one moved to bit 31 (exact for lz >= 1; for lz = 0, m's
    // last bit, a one, falls below bit 0 and `half` keeps it): f = (x + half/2) 2^-31
    const uint32_t x = (w << (lz & 31)) | (lz ? 1u << ((lz - 1) & 31) : 0u);
    const int32_t half = lz == 0 ? 1 : 0;
    const bool big = x >= 0xC0000000u;          // f >= 1.5: use f/2
    n = lz + (big ? 0 : 1);
    const int sh = big ? 21 : 20;
    J = (x >> sh) + ((x >> (sh - 1)) & 1u);
    // f' - c = (2 (x - J 2^sh) + half) 2^-(32 + big), an integer below 2^22 in magnitude
    const int32_t D = (int32_t)(x - (J << sh));
    return __int2float_rn(2 * D + half) * (big ? 0x1p-33f : 0x1p-32f);
}

// -2 ln((w + 1/2) 2^-32) of two words in double-float.
__device__ __forceinline__ FFP ff_neg2log2(uint32_t wa, uint32_t wb, const FFTables &t) {
    uint32_t Ja, Jb;
    int na, nb;
    const float da = ff_log_split(wa, Ja, na), db = ff_log_split(wb, Jb, nb);
    const float2 dk = make_float2(da, db);
    const float4 La = t.lg[Ja - (uint32_t)kLogFirst], Lb = t.lg[Jb - (uint32_t)kLogFirst];
    const float2 ch = make_float2(La.x, Lb.x), cl = make_float2(La.y, Lb.y);
    // r = (f' - c) / c
    const float2 rh = p_mul(dk, ch);
    const float2 rl = p_fma(dk, cl, p_fma(dk, ch, p_neg(rh)));
    // B = -2 ln(1 + r) = -2r + r^2 - r^3 (2/3 - r/2 + 2r^2/5): -2rh + rh^2 by the fast
    // two-sum (|2 rh| >= rh^2), the rest in single precision
    const float2 p = p_mul(rh, rh);
    const float2 pe = p_fma(rh, rh, p_neg(p));
    const float2 tail = p_mul(p_mul(p, rh), p_fma(rh, p_fma(rh, p2(-0.4f), p2(0.5f)), p2(-2.0f / 3.0f)));
    const float2 bh = p_fma(p2(-2.0f), rh, p);
    const float2 be = p_sub(p, p_fma(p2(2.0f), rh, bh));
    const float2 bl = p_add(p_add(p_fma(p2(-2.0f), rl, be), p_fma(p_mul(p2(2.0f), rh), rl, pe)), tail);
    // -2 ln c + B: |-2 ln c| >= 9.7e-4 > |B| unless c = 1 (then -2 ln c = 0); then
    // 2 n ln 2 + (..): 2 n ln 2 >= 1.38 > 0.82 unless n = 0
    const FFP X = p_add_ordered(FFP{make_float2(La.z, Lb.z), make_float2(La.w, Lb.w)}, FFP{bh, bl});
    const float2 Aa = t.ln2[na], Ab = t.ln2[nb];
    return p_add_ordered(FFP{make_float2(Aa.x, Ab.x), make_float2(Aa.y, Ab.y)}, X);
}

// sqrt(L) of two normalised double-floats 2^-33 < L < 64.
__device__ __forceinline__ FFP ff_sqrt2(FFP L) {
    const float2 y = make_float2(rsqrtf(L.hi.x), rsqrtf(L.hi.y));
    const float2 s0 = p_mul(L.hi, y);
    const float2 hy = p_mul(p2(0.5f), y);
    const float2 p = p_mul(s0, s0), pe = p_fma(s0, s0, p_neg(p));
    const float2 r0 = p_add(p_sub(p_sub(L.hi, p), pe), L.lo);              // L - s0^2
    const float2 c1 = p_mul(r0, hy);
    const float2 r1 = p_fma(p_neg(c1), c1, p_fma(p_mul(p2(-2.0f), s0), c1, r0));  // L - (s0 + c1)^2
    const FFP s = p_fast_two_sum(s0, c1);
    return FFP{s.hi, p_fma(r1, hy, s.lo)};
}

// The binary angle 2 pi (2w + 1) / 2^33 split into an octant o, a table angle a of the first
// octant (its double-float sine and cosine in tv) and the remainder's multiple rf of
// 2 pi / 2^33, taken with the sign that makes theta = (octant symmetry)(a + d).
__device__ __forceinline__ float ff_turn_split(uint32_t w, const FFTables &t, uint32_t &o, float4 &tv) {
    const uint32_t q = (w >> 20) + ((w >> 19) & 1u);        // nearest multiple of 2^21 of 2w + 1
    const int32_t rho = (int32_t)(2u * w + 1u - (q << 21));  // |rho| < 2^20, exact in float
    const uint32_t j = q & 4095u, m = j & 511u;
    o = j >> 9;
    const bool odd = o & 1u;                                 // reflected octant: a = pi/4 - ..
    tv = t.trig[odd ? 512u - m : m];
    return __int2float_rn(odd ? -rho : rho);
}

// Of two remainders d: sin d = dh + sdl, cos d - 1 = cmh + cml.
struct FFTurn2 {
    float2 dh, sdl, cmh, cml;
};
__device__ __forceinline__ FFTurn2 ff_turn2(float2 rf) {
    constexpr double C = 6.283185307179586 / 8589934592.0;  // 2 pi / 2^33
    constexpr float Ch = (float)C;
    constexpr float Cl = (float)(C - (double)Ch);
    FFTurn2 r;
    r.dh = p_mul(rf, p2(Ch));
    const float2 dl = p_fma(rf, p2(Cl), p_fma(rf, p2(Ch), p_neg(r.dh)));
    const float2 p = p_mul(r.dh, r.dh), pl = p_fma(r.dh, r.dh, p_neg(p)), nd = p_neg(r.dh);
    r.cmh = p_mul(p2(-0.5f), p);
    r.cml = p_fma(nd, dl, p_fma(p, p_mul(p, p2(1.0f / 24.0f)), p_mul(p2(-0.5f), pl)));
    r.sdl = p_fma(nd, p_mul(p, p2(1.0f / 6.0f)), dl);
    return r;
}

// P (1 + (cos d - 1)) + Q sin d for table values P, Q (double-float): sin(a + d) with
// (P, Q) = (sin a, cos a), cos(a + d) with (cos a, -sin a).
__device__ __forceinline__ FFP ff_rot2(float2 Ph, float2 Pl, float2 Qh, float2 Ql, float2 dh, float2 sdl, float2 cmh,
                                       float2 cml) {
    const float2 x = p_mul(Qh, dh), xl = p_fma(Qh, dh, p_neg(x));
    const float2 y = p_mul(Ph, cmh), yl = p_fma(Ph, cmh, p_neg(y));
    const FFP d = p_two_sum(x, y);
    const float2 small = p_fma(Qh, sdl, p_fma(Ql, dh, p_fma(Ph, cml, p_mul(Pl, cmh))));
    const float2 dl = p_add(p_add(d.lo, p_add(xl, yl)), small);
    const FFP s = p_two_sum(Ph, d.hi);
    return p_fast_two_sum(s.hi, p_add(s.lo, p_add(Pl, dl)));
}
__device__ __forceinline__ FF ff_rot(float Ph, float Pl, float Qh, float Ql, float dh, float sdl, float cmh,
                                     float cml) {
    const FF x = ff_two_prod(Qh, dh);
    const FF y = ff_two_prod(Ph, cmh);
    const FF d = ff_two_sum(x.hi, y.hi);
    const float small = fmaf(Qh, sdl, fmaf(Ql, dh, fmaf(Ph, cml, __fmul_rn(Pl, cmh))));
    const float dl = __fadd_rn(__fadd_rn(d.lo, __fadd_rn(x.lo, y.lo)), small);
    const FF s = ff_two_sum(Ph, d.hi);
    return ff_fast_two_sum(s.hi, __fadd_rn(s.lo, __fadd_rn(Pl, dl)));
}

// R V rounded to float with the rounding's error e = (R V) - f and the bound on the error of
// R V; ff_certain: the value lies outside the bound of the midpoints next to f (and f is no power
// of two, whose lower neighbour is half as far).
__device__ __forceinline__ bool ff_certain(float f, float e, float bound) {
    const uint32_t fb = __float_as_uint(f);
    const float half_ulp = __uint_as_float((fb & 0x7F800000u) - (24u << 23));
    return (fb & 0x7FFFFFu) != 0u && fabsf(e) + bound < half_ulp;
}

// The double-float factors of a Philox block's three Gaussians: R1 (cos, sin) of the first angle,
// R2 cos of the second.
struct FFFactors {
    FFP R;     // (R1, R2)
    FFP V;     // (cos, sin) of the first angle
    FF C2;     // cos of the second
};
__device__ __forceinline__ FFFactors ff_factors(const Philox4 &w, const FFTables &t) {
    FFFactors r;
    r.R = ff_sqrt2(ff_neg2log2(w.w0, w.w2, t));
    uint32_t oa, ob;
    float4 ta, tb;  // (sin hi, cos hi, sin lo, cos lo)
    const float ra = ff_turn_split(w.w1, t, oa, ta), rb = ff_turn_split(w.w3, t, ob, tb);
    const FFTurn2 d = ff_turn2(make_float2(ra, rb));
    // (sin, cos)(a + d) side by side
    const FFP sc = ff_rot2(make_float2(ta.x, ta.y), make_float2(ta.z, ta.w), make_float2(ta.y, -ta.x),
                           make_float2(ta.w, -ta.z), p2(d.dh.x), p2(d.sdl.x), p2(d.cmh.x), p2(d.cml.x));
    // octant o: (sin, cos) = (s, c), (c, s), (c, -s), (s, -c), (-s, -c), (-c, -s), (-c, s), (-s, c)
    const bool swap = ((oa + 1u) >> 1) & 1u;
    const uint32_t ns = (oa & 4u) << 29, nc = ((oa + 2u) & 4u) << 29;  // sign bits of the sine, the cosine
    auto flip = [](float v, uint32_t sign) { return __uint_as_float(__float_as_uint(v) ^ sign); };
    r.V.hi = make_float2(flip(swap ? sc.hi.x : sc.hi.y, nc), flip(swap ? sc.hi.y : sc.hi.x, ns));
    r.V.lo = make_float2(flip(swap ? sc.lo.x : sc.lo.y, nc), flip(swap ? sc.lo.y : sc.lo.x, ns));
    const bool swap2 = ((ob + 1u) >> 1) & 1u;
    const FF c2 = ff_rot(swap2 ? tb.x : tb.y, swap2 ? tb.z : tb.w, swap2 ? tb.y : -tb.x, swap2 ? tb.w : -tb.z, d.dh.y,
                         d.sdl.y, d.cmh.y, d.cml.y);
    const uint32_t nc2 = ((ob + 2u) & 4u) << 29;
    r.C2 = FF{flip(c2.hi, nc2), flip(c2.lo, nc2)};
    return r;
}

// Three standard Gaussians of one Philox block rounded to float (the values of box_muller3
// rounded to nearest); false when a rounding is not certain, and the caller must then take
// the FP64 transform's rounded values instead.
__device__ __forceinline__ bool box_muller3_ff(const Philox4 &w, const FFTables &t, float &g0, float &g1,
                                               float &g2) {
    const FFFactors q = ff_factors(w, t);
    const float2 Rh = p2(q.R.hi.x), Rl = p2(q.R.lo.x);
    const float2 gh = p_mul(Rh, q.V.hi);
    const float2 ge = p_add(p_fma(Rh, q.V.hi, p_neg(gh)), p_fma(Rh, q.V.lo, p_mul(Rl, q.V.hi)));
    const float2 f = p_add(gh, ge);
    const float2 e = p_add(p_sub(gh, f), ge);  // (gh + ge) - f
    const float hh = __fmul_rn(q.R.hi.y, q.C2.hi);
    const float he = __fadd_rn(fmaf(q.R.hi.y, q.C2.hi, -hh), fmaf(q.R.hi.y, q.C2.lo, __fmul_rn(q.R.lo.y, q.C2.hi)));
    const float h = __fadd_rn(hh, he);
    const float e2 = __fadd_rn(__fsub_rn(hh, h), he);
    g0 = f.x;
    g1 = f.y;
    g2 = h;
    const float2 rb = p_mul(q.R.hi, p2(0x1p-43f));
    return ff_certain(f.x, e.x, fmaf(fabsf(f.x), 0x1p-41f, rb.x)) &&
           ff_certain(f.y, e.y, fmaf(fabsf(f.y), 0x1p-41f, rb.x)) &&
           ff_certain(h, e2, fmaf(fabsf(h), 0x1p-41f, rb.y));
}

// The FP64 transform's Gaussians rounded to float (reading the FP64 tables from global
// memory): the rare draws whose double-float rounding is not certain.
static __device__ __noinline__ void box_muller3_fp64_rounded(Philox4 w, const double2 *tab, float *g) {
    const SmemTables &t = *reinterpret_cast<const SmemTables *>(tab);
    double d0, d1, d2;
    box_muller3(w, t, d0, d1, d2);
    g[0] = d2f_bits(d0);
    g[1] = d2f_bits(d1);
    g[2] = d2f_bits(d2);
}

// Three standard Gaussians rounded to float: the FP64 transform's values, bit for bit.
__device__ __forceinline__ void gaussians_f32(const Philox4 &w, const FFTables &t, const double2 *tab64, float &g0,
                                              float &g1, float &g2) {
    if (!box_muller3_ff(w, t, g0, g1, g2)) {
        float g[3];
        box_muller3_fp64_rounded(w, tab64, g);
        g0 = g[0];
        g1 = g[1];
        g2 = g[2];
    }
}

}  // namespace ss
