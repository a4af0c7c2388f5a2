// wide_math.cuh -- FP64 results of the FP64-state particle pass computed on the FP32 and
// integer pipes, bit for bit.
//
// GB300 issues two FP64 instructions per clock and SM against 128 FP32 or integer ones, so
// an FP64 instruction costs as much as 64 others.  The functions here give the bits of
// an FP64 formula without its FP64 instructions: each forms the formula's last, rounded
// value with some bits to spare and a bound on its distance from what FP64 arithmetic
// gets; where that value lies so near a rounding boundary that the bound could cross it
// (one evaluation in 2^11 or rarer), it says so and the caller runs the FP64 formula.
//   w_rsqrt53: rsqrt_fp64's four FP64 instructions (~50 others), w_square53 its square (~20),
//              w_mul53 its product with a double;
//   w_add:     the sum of a double and a much smaller float (~25, and no conversion);
//   w_kick:    the kick's integrals as the FP32 values their user reads (9 FP64
//              instructions as polynomials, 8 per node as sums);
//   w_sqrt53, w_div53: correctly rounded roots and quotients (the sampler, |q|, the weights).
// tests/test_wide_math.py compares them with the FP64 formulas, bit for bit.
//
// Plain C++ besides the intrinsics, so that the test compiles it for the host.
#pragma once

#include <cstdint>

namespace fdf {

#define FDF_DEV __device__ __forceinline__

// ---- rsqrt_fp64 (device_math.cuh) in integers -------------------------------------------
// For v in the FP32 normal range and its FP32 estimate yf = rsqrtf(d2f_bits(v)), the bits of
//   r = fma(y, s, y),  s = eh + 1.5f eh^2,  eh = fma(-(v y), y/2, 0.5)
// v = m 4^k with 1 <= m < 4 and y = h 2^-k: every operation scales exactly, so m and h
// serve as integers M 2^-52 and Y 2^-24 (54 and 24 bits).  m h is rounded to 53 bits as
// FP64 rounds it; eh is exact (FP64 drops at most two of its bits); the FP32 term 1.5f eh^2
// is formed in FP32 as well; h s and the final sum are exact to 2^-69.  What FP64 rounds
// differently before the final rounding (eh and s below 2^-76, the FP32 square below
// 2^-66) amounts to less than 12 of these units; the final rounding is at 2^-53, so a
// value within 16 units of a tie (33 of 65536) is left to FP64, as is one whose
// intermediate values leave the binades assumed (m within 2^-20 of 1 or 4).
// R and k: r = R 2^(-53 - k).
FDF_DEV bool w_rsqrt53(double v, float yf, double& r, int64_t& R, int& k)
{
    const uint32_t hi = (uint32_t)__double2hiint(v), lo = (uint32_t)__double2loint(v);
    const int ex = (int)(hi >> 20) - 1023, odd = ex & 1;
    k = ex >> 1;
    const uint32_t m1 = (hi & 0xFFFFFu) | 0x100000u;
    const uint32_t Mh = odd ? (m1 << 1) | (lo >> 31) : m1, Ml = lo << odd;
    const uint32_t yb = __float_as_uint(yf);
    const uint32_t Y = (yb & 0x7FFFFFu) | 0x800000u;
    bool ok = hi - 0x38100000u < 0x0FE00000u;                    // v in the FP32 normal range
    ok = ok && (int)(yb >> 23) + k == 126;                       // 1/2 <= h < 1
    // V = m h in units of 2^-52, rounded to nearest, ties to even
    const uint64_t a = (uint64_t)Ml * Y;
    const uint64_t b = (uint64_t)Mh * Y + (a >> 32);
    const uint32_t al = (uint32_t)a, bl = (uint32_t)b, bh = (uint32_t)(b >> 32);
    uint64_t V = ((uint64_t)__funnelshift_l(bl, bh, 8) << 32) | __funnelshift_l(al, bl, 8);
    V += (al >> 23) & (uint32_t)((al & 0x7FFFFFu) != 0u || (V & 1u));
    const uint32_t Vh = (uint32_t)(V >> 32), Vl = (uint32_t)V;
    ok = ok && (Vh >> 20) == 1u;                                 // 1 <= m h < 2
    // E = 1/2 - V h / 2 in units of 2^-77 (the low 64 bits hold it)
    const int64_t E = -(int64_t)((uint64_t)Vl * Y + ((uint64_t)(Vh * Y) << 32));
    const float eh = __fmul_rn(__int2float_rn((int)(E >> 25)), 2.220446049250313081e-16f);   // 2^-52
    const float kap = __fmul_rn(__fmul_rn(1.5f, eh), eh);
    // h (E + kap) in units of 2^-69
    const float h69 = __fmul_rn(__uint2float_rn(Y), 35184372088832.f);                       // h 2^69
    const int64_t W = (int64_t)(int)Y * (int)(E >> 32) + (int64_t)(((uint64_t)(uint32_t)E * Y) >> 32) +
                      __float2int_rn(__fmul_rn(kap, h69));
    ok = ok && ((uint32_t)W & 0xFFFFu) - (0x8000u - 16u) > 32u;
    R = ((int64_t)Y << 29) + ((W + 0x8000) >> 16); // r 2^k in units of 2^-53
    const uint32_t Rh = (uint32_t)(R >> 32);
    ok = ok && (Rh >> 20) == 1u;
    r = __hiloint2double((int)(Rh + ((uint32_t)(1021 - k) << 20)), (int)(uint32_t)R);
    return ok;
}

FDF_DEV bool w_rsqrt53(double v, float yf, double& r)
{
    int64_t R;
    int k;
    return w_rsqrt53(v, yf, r, R, k);
}

// The bits of r * r for r = R 2^(-53 - k), 2^52 <= R < 2^53 (w_rsqrt53's), rounded to nearest,
// ties to even: the 106-bit square in three 32-bit products.
FDF_DEV double w_square53(int64_t R, int k)
{
    const uint32_t Rh = (uint32_t)((uint64_t)R >> 32), Rl = (uint32_t)R;
    const uint64_t ll = (uint64_t)Rl * Rl;
    const uint64_t mid = (((uint64_t)Rh * Rl) << 1) + (ll >> 32);
    const uint64_t top = (uint64_t)Rh * Rh + (mid >> 32);       // the square's bits 64 ..
    const uint32_t m = (uint32_t)mid, th = (uint32_t)(top >> 32), tl = (uint32_t)top;
    const uint32_t big = th >> 9;                               // the square >= 2^105
    const uint32_t sh = 12u - big;
    const uint32_t ql = __funnelshift_l(m, tl, sh), rem = m << sh;
    const uint32_t sticky = ((uint32_t)ll != 0u) | (ql & 1u);
    const uint64_t q = (((uint64_t)__funnelshift_l(tl, th, sh) << 32) | ql) + (rem > 0x80000000u - sticky);
    return __hiloint2double((int)((uint32_t)(q >> 32) + ((1020u + big - 2u * (uint32_t)k) << 20)), (int)(uint32_t)q);
}

// The bits of r * g for r as above, rounded to nearest, ties to even, from the 106-bit product;
// false unless g and the product are finite normal numbers.
FDF_DEV bool w_mul53(int64_t R, int k, double g, double& x)
{
    const uint32_t Rh = (uint32_t)((uint64_t)R >> 32), Rl = (uint32_t)R;
    const uint32_t gh = (uint32_t)__double2hiint(g), Gl = (uint32_t)__double2loint(g);
    const uint32_t Gh = (gh & 0xFFFFFu) | 0x100000u;
    const int eg = (int)((gh >> 20) & 0x7FFu);
    const uint64_t ll = (uint64_t)Rl * Gl;
    const uint64_t m1 = (uint64_t)Rh * Gl + (ll >> 32);
    const uint64_t m2 = (uint64_t)Rl * Gh + (uint32_t)m1;
    const uint64_t top = (uint64_t)Rh * Gh + (m1 >> 32) + (m2 >> 32);
    const uint32_t m = (uint32_t)m2, th = (uint32_t)(top >> 32), tl = (uint32_t)top;
    const uint32_t big = th >> 9;                               // the product of significands >= 2^105
    const uint32_t sh = 12u - big;
    const uint32_t ql = __funnelshift_l(m, tl, sh), rem = m << sh;
    const uint32_t sticky = ((uint32_t)ll != 0u) | (ql & 1u);
    const uint64_t q = (((uint64_t)__funnelshift_l(tl, th, sh) << 32) | ql) + (rem > 0x80000000u - sticky);
    // r's exponent is -1 - k, so the product's is eg - 1 - k, or one less
    const int e = eg - 2 + (int)big - k;
    x = __hiloint2double((int)(((uint32_t)(q >> 32) + ((uint32_t)e << 20)) | (gh & 0x80000000u)), (int)(uint32_t)q);
    return (unsigned)(eg - 1) < 0x7FEu && e >= 0 && e < 0x7FD;
}

// The bits of q + (double)d in integers (a subnormal d counts as zero, as f2d_bits takes it):
// d's 24-bit significand in units of q's last place, rounded to nearest, ties to even, is
// added to q's bit pattern.  False where that may not be the sum's pattern: the sum leaves q's
// binade or comes to its lower end (below which last places are finer), |d| is above 2^-1 |q|
// or so, or one of them is no finite normal number.
FDF_DEV bool w_add(double q, float d, double& r)
{
    const uint32_t hi = (uint32_t)__double2hiint(q), lo = (uint32_t)__double2loint(q), db = __float_as_uint(d);
    const int eq = (int)((hi >> 20) & 0x7FFu), ed = (int)((db >> 23) & 0xFFu);
    const int F = ed ? (int)((db & 0x7FFFFFu) | 0x800000u) : 0;
    const int Z = (int)(db ^ hi) < 0 ? -F : F;
    const int s = eq - ed - 925;                                // d = Z 2^-s in units of q's last place
    const int S = s > 31 ? 31 : (s > 0 ? s : 0), L = s < 0 ? -s : 0;
    const uint32_t below = __funnelshift_r(0u, (uint32_t)Z, (uint32_t)S);    // the bits that go, at the top of a word
    int X = Z >> S;
    X += below > 0x80000000u - ((lo + (uint32_t)X) & 1u);
    const uint64_t delta = ((uint64_t)(uint32_t)(int)__funnelshift_l((uint32_t)X, (uint32_t)(X >> 31), (uint32_t)L) << 32) |
                           ((uint32_t)X << (L & 31));
    const uint64_t b = (((uint64_t)hi << 32) | lo) + delta;
    const uint32_t bh = (uint32_t)(b >> 32);
    r = __hiloint2double((int)bh, (int)(uint32_t)b);
    return L <= 27 && ed != 255 && (uint32_t)(eq - 1) < 0x7FEu && ((bh ^ hi) >> 20) == 0u &&
           ((bh & 0xFFFFFu) | (uint32_t)b) != 0u;
}

// ---- correctly rounded root and quotient ------------------------------------------------
// An estimate within a few last places, its exact remainder modulo 2^64 (the remainder is
// small, so the low 64 bits hold it), the correction that the remainder asks for, and a test
// of the corrected remainder that no other 53-bit number is nearer: the IEEE result
// whatever the estimate's error, or false.

// sqrt(u) from the FP32 estimate yf = rsqrtf(d2f_bits(u)): u = M 2^-52 4^k and the root
// S 2^(k-52), 2^52 <= S < 2^53, where S^2 is nearest M 2^52.
FDF_DEV bool w_sqrt53(double u, float yf, double& root)
{
    const uint32_t hi = (uint32_t)__double2hiint(u), lo = (uint32_t)__double2loint(u);
    const int ex = (int)(hi >> 20) - 1023, k = ex >> 1, odd = ex & 1;
    const uint32_t m1 = (hi & 0xFFFFFu) | 0x100000u;
    const uint32_t Mh = odd ? (m1 << 1) | (lo >> 31) : m1, Ml = lo << odd;
    const uint32_t yb = __float_as_uint(yf);
    const uint32_t Y = (yb & 0x7FFFFFu) | 0x800000u;
    bool ok = hi - 0x38100000u < 0x0FE00000u && (int)(yb >> 23) + k == 126;
    // V = m h and E = (1 - V h) / 2 as in w_rsqrt53; the root is V (1 + 2 E / 2 ...): V + V E
    const uint64_t a = (uint64_t)Ml * Y;
    const uint64_t b = (uint64_t)Mh * Y + (a >> 32);
    const uint32_t al = (uint32_t)a, bl = (uint32_t)b, bh = (uint32_t)(b >> 32);
    const uint64_t V = ((uint64_t)__funnelshift_l(bl, bh, 8) << 32) | __funnelshift_l(al, bl, 8);
    const uint32_t Vh = (uint32_t)(V >> 32), Vl = (uint32_t)V;
    const int64_t E = -(int64_t)((uint64_t)Vl * Y + ((uint64_t)(Vh * Y) << 32));     // units of 2^-77
    // V (E + 3 E^2 / 2) in units of 2^-52
    const float eh = __fmul_rn(__int2float_rn((int)(E >> 25)), 2.220446049250313081e-16f);     // 2^-52
    const float kap = __fmul_rn(__fmul_rn(1.5f, eh), eh);
    const int64_t step = (((int64_t)(int)(V >> 22) * (int)(E >> 25)) >> 30) +
                         __float2int_rn(__fmul_rn(__fmul_rn(kap, __uint2float_rn(Vh)), 4294967296.f));
    const uint64_t S0 = V + (uint64_t)step;
    const uint32_t Sl = (uint32_t)S0, Sh = (uint32_t)(S0 >> 32);
    int64_t rem = (int64_t)(((uint64_t)Ml << 52) - ((uint64_t)Sl * Sl + ((uint64_t)(2u * Sl * Sh) << 32)));
    // n = rem / (2 S), 1 / (2 S) = h 2^-53
    const int n = __float2int_rn(__fmul_rn(__fmul_rn(__int2float_rn((int)(rem >> 32)), __uint2float_rn(Y)),
                                           2.842170943040401e-14f));                           // 2^(32 - 53 - 24)
    const int64_t S = (int64_t)S0 + n;
    rem -= n * ((int64_t)S0 + S);
    ok = ok && rem <= S && rem > -S && (uint32_t)((uint64_t)S >> 52) == 1u;
    root = __hiloint2double((int)((uint32_t)((uint64_t)S >> 32) + ((uint32_t)(1022 + k) << 20)), (int)(uint32_t)S);
    return ok;
}

// a / b from an estimate q within a few last places.
FDF_DEV bool w_div53(double a, double b, double q, double& r)
{
    const uint32_t ah = (uint32_t)__double2hiint(a), bh = (uint32_t)__double2hiint(b), qh = (uint32_t)__double2hiint(q);
    const int ea = (int)((ah >> 20) & 0x7FFu), eb = (int)((bh >> 20) & 0x7FFu), eq = (int)((qh >> 20) & 0x7FFu);
    const uint64_t A = ((uint64_t)((ah & 0xFFFFFu) | 0x100000u) << 32) | (uint32_t)__double2loint(a);
    const uint32_t Bh = (bh & 0xFFFFFu) | 0x100000u, Bl = (uint32_t)__double2loint(b);
    const uint64_t B = ((uint64_t)Bh << 32) | Bl;
    const uint32_t Qh = (qh & 0xFFFFFu) | 0x100000u, Ql = (uint32_t)__double2loint(q);
    // the remainder A 2^s - Q B, s = 52 or 53
    const int sft = ea - eb - eq + 1075;
    bool ok = (unsigned)(ea - 1) < 0x7FEu && (unsigned)(eb - 1) < 0x7FEu && (unsigned)(eq - 1) < 0x7FEu &&
              (sft == 52 || sft == 53) && (int)(ah ^ bh ^ qh) >= 0;
    int64_t rem = (int64_t)((A << (sft & 63)) - ((uint64_t)Ql * Bl + ((uint64_t)(Qh * Bl + Ql * Bh) << 32)));
    // n = rem / B, B = f 2^52
    const float f = __uint_as_float(0x3F800000u | ((Bh & 0xFFFFFu) << 3) | (Bl >> 29));
    const int n = __float2int_rn(__fmul_rn(__fmul_rn(__int2float_rn((int)(rem >> 32)), 9.5367431640625e-7f), w_rcp(f)));
    rem -= (int64_t)n * (int64_t)B;
    const uint64_t bits = (((uint64_t)qh << 32) | Ql) + (uint64_t)(int64_t)n;
    ok = ok && 2 * rem <= (int64_t)B && 2 * rem >= -(int64_t)B && (((uint32_t)(bits >> 32) ^ qh) >> 20) == 0u &&
         (((uint32_t)(bits >> 32) << 12) | (uint32_t)bits) != 0u;
    r = __hiloint2double((int)(uint32_t)(bits >> 32), (int)(uint32_t)bits);
    return ok;
}

// (float)d and (double)f in integers: the bits of the plain casts for every value.  What lies
// outside FP32's normal range (zeros, subnormals, overflows, infinities, NaN) is left to the
// cast itself, as a call: inlined, every argument would run its FP64 instruction.
static __device__ __attribute__((noinline)) float w_d2f_rest(double d) { return (float)d; }
static __device__ __attribute__((noinline)) double w_f2d_rest(float f) { return (double)f; }

FDF_DEV float w_d2f(double d)
{
    const uint32_t hi = (uint32_t)__double2hiint(d), lo = (uint32_t)__double2loint(d);
    const uint32_t mag = hi & 0x7FFFFFFFu;
    uint32_t f = ((mag - 0x38000000u) << 3) | (lo >> 29);
    f += (lo & 0x1FFFFFFFu) > 0x10000000u - (f & 1u);
    float r = __uint_as_float((hi & 0x80000000u) | f);
    if (mag - 0x38100000u >= 0x0FE00000u) r = w_d2f_rest(d);
    return r;
}

FDF_DEV double w_f2d(float f)
{
    const uint32_t b = __float_as_uint(f), mag = b & 0x7FFFFFFFu;
    double r = __hiloint2double((int)(((mag >> 3) + 0x38000000u) | (b & 0x80000000u)), (int)(b << 29));
    if (mag - 0x00800000u >= 0x7F000000u) r = w_f2d_rest(f);
    return r;
}

// ---- pairs of floats (value = hi + lo, 48 bits) -----------------------------------------
FDF_DEV void w_two_sum(float a, float b, float& s, float& e)
{
    s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}

// (sh, sl) = c + t (sh, sl)
FDF_DEV void w_horner(float ch, float cl, float th, float tl, float& sh, float& sl)
{
    const float p = __fmul_rn(th, sh);
    float e = __fmaf_rn(th, sh, -p);
    e = __fmaf_rn(th, sl, e);
    e = __fmaf_rn(tl, sh, e);
    float l;
    w_two_sum(ch, p, sh, l);
    sl = __fadd_rn(l, __fadd_rn(cl, e));
}

// ---- the kick's integrals ---------------------------------------------------------------
// Polynomials in t = m^2 a_c^2 / u_0 (WideCoef says of what), coefficients h[k] + l[k].
constexpr int kKickDeg = 10;    // highest degree
// SERIES: the pass's fitted polynomials (c_0 in FP64, the others FP32), evaluated as the
// FP64 formula does: u^(-1/2) to first order, t and the terms above c_0 in FP32.  Up to degree
// 5, which steps of d ln a up to 0.111 need (155 steps from z = 1e9 to 31 and more).
// !SERIES: the sums over the nodes themselves, from polynomials that agree with them to
// 2^-47 (wide_poly.cuh); c_1 .. c_6 as pairs.
template <bool SERIES> struct KickLen {
    static constexpr int kDeg = SERIES ? 5 : 10;
    static constexpr int kPair = SERIES ? 1 : 7;
};
struct KickPoly {
    float h[kKickDeg + 1], l[kKickDeg + 1];
};

// K_psi = u_0^(1/2) psi(t) and K_phi = u_0^(-1/2) phi(t) as FP32, u_0 = s_0 + mu, s_0 = |q_0|^2
// and mu = m^2 a_c^2 as pairs in the run's momentum unit.  A result that +-2^-41 does not move to another float counts as
// FP64's (rounded to FP32).  The margin is a choice, not a derived bound: pairs carry about
// 2^-44 of the result and FP64's own error is below 2^-50, and no result so accepted had other
// bits than the FP64 formula's, on the host (tests/test_wide_math.py) and in whole runs on the
// device (tests/test_gpu_wide_bits.py).  Returns whether both are.
template <bool SERIES>
FDF_DEV bool w_kick(float s0h, float s0l, float muh, float mul, const KickPoly& psi, const KickPoly& phi, float& Kpsi,
                    float& Kphi)
{
    float uh, ul;
    w_two_sum(s0h, muh, uh, ul);
    ul = __fadd_rn(ul, __fadd_rn(s0l, mul));
    const float y = w_rsqrt(uh);
    const float y2 = __fmul_rn(y, y), y2e = __fmaf_rn(y, y, -y2);
    float e = __fmaf_rn(-uh, y2, 1.f);
    e = __fmaf_rn(-uh, y2e, e);
    e = __fmaf_rn(-ul, y2, e);
    // u^(-1/2) = y (1 + c)
    const float c = SERIES ? __fmul_rn(0.5f, e) : __fmul_rn(e, __fmaf_rn(0.375f, e, 0.5f));
    bool ok = true;
    float t, tl = 0.f;
    if (SERIES) {
        const float r = __fmaf_rn(y, c, y);
        ok = __fmaf_rn(y, __fadd_rn(c, 2.2737368e-13f), y) == __fmaf_rn(y, __fsub_rn(c, 2.2737368e-13f), y);  // 2^-42
        t = __fmul_rn(__fmul_rn(muh, r), r);
    } else {
        t = __fmul_rn(muh, y2);
        tl = __fmaf_rn(muh, y2, -t);
        tl = __fmaf_rn(muh, y2e, tl);
        tl = __fmaf_rn(mul, y2, tl);
        tl = __fmaf_rn(t, __fmaf_rn(e, e, e), tl);
    }
    constexpr int DEG = KickLen<SERIES>::kDeg, PAIR = KickLen<SERIES>::kPair;
    float a = phi.h[DEG], b = psi.h[DEG], a1 = 0.f, b1 = 0.f;
#pragma unroll
    for (int k = DEG - 1; k >= PAIR; --k) {
        a = __fmaf_rn(a, t, phi.h[k]);
        b = __fmaf_rn(b, t, psi.h[k]);
    }
#pragma unroll
    for (int k = PAIR - 1; k >= 1; --k) {
        w_horner(phi.h[k], phi.l[k], t, tl, a, a1);
        w_horner(psi.h[k], psi.l[k], t, tl, b, b1);
    }
    const float pa = __fmul_rn(a, t), pb = __fmul_rn(b, t);
    float qa = __fmaf_rn(a, t, -pa), qb = __fmaf_rn(b, t, -pb);
    if (!SERIES) {
        qa = __fmaf_rn(a1, t, __fmaf_rn(a, tl, qa));
        qb = __fmaf_rn(b1, t, __fmaf_rn(b, tl, qb));
    }
    const float ah = __fadd_rn(phi.h[0], pa), bh = __fadd_rn(psi.h[0], pb);
    const float al = __fadd_rn(__fsub_rn(pa, __fsub_rn(ah, phi.h[0])), __fadd_rn(phi.l[0], qa));
    const float bl = __fadd_rn(__fsub_rn(pb, __fsub_rn(bh, psi.h[0])), __fadd_rn(psi.l[0], qb));
    // K_phi = y (1 + c) (ah + al)
    float h = __fmul_rn(y, ah);
    float l = __fmaf_rn(y, __fmaf_rn(ah, c, al), __fmaf_rn(y, ah, -h));
    float d = __fmul_rn(h, 4.5474735e-13f);                      // 2^-41
    Kphi = __fadd_rn(h, __fadd_rn(l, d));
    ok = ok && Kphi == __fadd_rn(h, __fsub_rn(l, d));
    // K_psi = u y (1 + c) (bh + bl)
    const float w = __fmul_rn(uh, y);
    float wl = __fmaf_rn(uh, y, -w);
    wl = __fmaf_rn(ul, y, wl);
    wl = __fmaf_rn(w, c, wl);
    h = __fmul_rn(w, bh);
    l = __fmaf_rn(w, bh, -h);
    l = __fmaf_rn(w, bl, l);
    l = __fmaf_rn(wl, bh, l);
    d = __fmul_rn(h, 4.5474735e-13f);
    Kpsi = __fadd_rn(h, __fadd_rn(l, d));
    return ok && Kpsi == __fadd_rn(h, __fsub_rn(l, d));
}

}  // namespace fdf
