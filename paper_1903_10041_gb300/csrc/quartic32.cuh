// Quartic minimiser for the mixed-precision solver: Algorithm 1 (Sec. III-B)
// evaluated in FP32, with every branch decision of the cubic taken as FP64
// would take it.
//
// Same mathematics as quartic64.cuh.  Differences:
//  * The sign of Delta = Q^3 + R^2 is computed in FP32 together with a
//    forward error bound (first-order propagation of one unit roundoff per
//    FP32 operation through b, c, d, Q, R and Delta, with a safety factor
//    of at least 1.25 on every term).  When |Delta| exceeds the bound the
//    FP32 sign is the exact sign, and therefore FP64's.  Otherwise b, c, d, Q, R
//    and Delta are recomputed in FP64 from the same A, B, C, D and the FP64
//    values decide the branch (and the Q = R = 0 test).
//  * The closed-form roots lose about log10(|b|/|x|) digits to cancellation
//    in FP32, so each candidate gets one Newton step on the derivative of
//    the original quartic, 4A x^3 + 3B x^2 + 2C x + D, which is evaluated
//    without that cancellation.  The step is taken
//    only where the quartic is convex (a minimiser) and the step is small,
//    so it cannot jump to another root.
//  * The two minima are compared through the factored difference
//    F(u) - F(v) = (u - v) [ (u^3 + u^2 v + u v^2 + v^3)/4 + (b/3)(u^2 + u v + v^2)
//                            + (c/2)(u + v) + d ],
//    which is the delta-f of Algorithm 1 without its cancellation.
#pragma once
#include "common.cuh"
#include "quartic64.cuh"

namespace admm_impl {

// Fast FP32 primitives for the closed forms: single special-function
// instructions that take denormals as zero (the forms that do not scale
// operand and result around each, three to four instructions more).  Their
// few-ulp errors are removed by the Newton step that follows (the root it
// converges to depends only on the coefficients), and the discriminant bound
// below allows for a reciprocal that is off by 2 ulp.  A denormal operand
// gives an infinity and one above 2^126 a zero.  Where a root is such a
// quotient itself (A = 0) or A's reciprocal left the range, the scalar code
// takes FP64 (rcp_in_range); elsewhere an infinity ends in a non-finite root or
// an uncertified discriminant, which go to FP64 too.
__device__ __forceinline__ float rcp_fast(float v)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(v));
    return r;
}
// Is r = rcp_fast(v) the reciprocal of a v > 0 (not flushed to an infinity or a zero)?
__device__ __forceinline__ bool rcp_in_range(float r) { return __float_as_uint(r) - 1u < 0x7f7fffffu; }
__device__ __forceinline__ float rsqrt_fast(float v)
{
    float r;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(v));
    return r;
}
__device__ __forceinline__ float sqrt_fast(float v) { return v > 0.0f ? v * rsqrt_fast(v) : 0.0f; }
// |v|^(1/3) for v != 0
__device__ __forceinline__ float cbrt_abs(float v)
{
    float l, r;
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(l) : "f"(fabsf(v)));
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(l * (1.0f / 3.0f)));
    return r;
}
__device__ __forceinline__ float cbrt_fast(float v) { return copysignf(v != 0.0f ? cbrt_abs(v) : 0.0f, v); }

// The FP64 closed form, out of line: taken only when FP32 overflows.
static __device__ __noinline__ float quartic_min_fallback64(float A, float B, float C, float D, float lo, float hi,
                                                     int paper_mode)
{
    return (float)quartic_min64((double)A, (double)B, (double)C, (double)D, (double)lo, (double)hi, paper_mode);
}

// One Horner step s <- s x + a with its rounding errors carried in c
// (compensated Horner scheme: error-free product by FMA, TwoSum for the
// addition; Graillat, Langlois and Louvet, 2005).
__device__ __forceinline__ void horner_comp_step(float &s, float &c, float x, float a)
{
    const float p = __fmul_rn(s, x);
    const float pe = __fmaf_rn(s, x, -p);
    const float t = __fadd_rn(p, a);
    const float bb = __fsub_rn(t, p);
    const float se = __fadd_rn(__fsub_rn(p, __fsub_rn(t, bb)), __fsub_rn(a, bb));
    s = t;
    c = __fmaf_rn(c, x, __fadd_rn(pe, se));
}

// Newton step on the quartic's derivative 4A x^3 + 3B x^2 + 2C x + D in
// FP32 Horner form.  Built with ADMM_COMPENSATED_POLISH, the derivative is
// evaluated by the compensated Horner scheme instead (about twice the
// working precision: the polished root is then the FP32 number nearest the
// root of the FP32 coefficients rather than up to a few units off it).
__device__ __forceinline__ float newton_polish32(float A, float B, float C, float D, float x)
{
#ifndef ADMM_COMPENSATED_POLISH
    // the operations and roundings of newton_polish32x2, lane for lane
    const float C2 = __fadd_rn(C, C);
    const float fp = __fmaf_rn(__fmaf_rn(__fmaf_rn(__fmul_rn(4.0f, A), x, __fmul_rn(3.0f, B)), x, C2), x, D);
    const float fpp = __fmaf_rn(__fmaf_rn(__fmul_rn(12.0f, A), x, __fmul_rn(6.0f, B)), x, C2);
    if (fpp > 0.0f) {
        const float dx = __fmul_rn(fp, rcp_fast(fpp));
        if (fabsf(dx) <= __fmul_rn(0.0625f, __fadd_rn(fabsf(x), 1.0f))) x = __fsub_rn(x, dx);
    }
    return x;
#else
    float s = 4.0f * A, c = 0.0f;
    horner_comp_step(s, c, x, 3.0f * B);
    horner_comp_step(s, c, x, 2.0f * C);
    horner_comp_step(s, c, x, D);
    const float fp = s + c;
    const float fpp = (12.0f * A * x + 6.0f * B) * x + 2.0f * C;
    if (fpp > 0.0f) {
        const float dx = fp * rcp_fast(fpp);
        if (fabsf(dx) <= 0.0625f * (fabsf(x) + 1.0f)) x -= dx;
    }
    return x;
#endif
}

// Sign of F(u) - F(v) via the factored form (F' = x^3 + b x^2 + c x + d).
__device__ __forceinline__ float delta_f32(float u, float v, float b, float c, float d)
{
    const float br = 0.25f * (u * u * u + u * u * v + u * v * v + v * v * v) +
                     (b * (1.0f / 3.0f)) * (u * u + u * v + v * v) + 0.5f * c * (u + v) + d;
    return (u - v) * br;
}

// FP64-cubic variant: b, c, d, Q, R, Delta, roots and delta-f in FP64.
__device__ __forceinline__ float quartic_min_fp64cubic(float A, float B, float C, float D, float lo, float hi,
                                                       int paper_mode)
{
    return (float)quartic_min64((double)A, (double)B, (double)C, (double)D, (double)lo, (double)hi, paper_mode);
}

// The branch of Algorithm 1 decided in FP64 from the same A, B, C, D.
static __device__ __noinline__ int cubic_branch64(float A, float B, float C, float D)
{
    const double inv64 = 1.0 / (double)A;
    const double bd = 0.75 * (double)B * inv64, cd = 0.5 * (double)C * inv64, dd = 0.25 * (double)D * inv64;
    const double b3d = bd * (1.0 / 3.0);
    const double Qd = cd * (1.0 / 3.0) - b3d * b3d;
    const double Rd = b3d * (0.5 * cd) - b3d * b3d * b3d - 0.5 * dd;
    const double Dd = Qd * Qd * Qd + Rd * Rd;
    return Dd > 0.0 ? 0 : ((Qd == 0.0 && Rd == 0.0) ? 1 : 2);
}

// FP32 variant with FP64-certified branch decisions.  `esc` counts the
// decisions that needed FP64.
__device__ __forceinline__ float quartic_min32(float A, float B, float C, float D, float lo, float hi,
                                               int paper_mode, unsigned &esc)
{
    if (A == 0.0f) {
        const float r = rcp_fast(__fadd_rn(C, C));
        if (!rcp_in_range(r)) return quartic_min_fallback64(A, B, C, D, lo, hi, paper_mode);
        return clampf(__fmul_rn(-D, r), lo, hi);
    }
    // unfused, so that an input near a double root or a tie keeps the rounding it always had
    const float inv = rcp_fast(A);
    const float b = __fmul_rn(__fmul_rn(0.75f, B), inv);
    const float c = __fmul_rn(__fmul_rn(0.5f, C), inv);
    const float d = __fmul_rn(__fmul_rn(0.25f, D), inv);
    const float b3 = __fmul_rn(b, 1.0f / 3.0f);
    const float b3s = __fmul_rn(b3, b3), b3c = __fmul_rn(b3s, b3);
    const float Q = __fmaf_rn(c, 1.0f / 3.0f, -b3s);
    const float bhc = __fmul_rn(b3, __fmul_rn(0.5f, c));
    const float R = __fsub_rn(__fsub_rn(bhc, b3c), __fmul_rn(0.5f, d));
    const float Qs = __fmul_rn(Q, Q);
    const float Dl = __fadd_rn(__fmul_rn(Qs, Q), __fmul_rn(R, R));
    // magnitudes entering Q, R (including the rounding of b, c, d); |Q| <= mQ and |R| <= mR
    const float mQ = __fmaf_rn(fabsf(c), 1.0f / 3.0f, b3s);
    const float mR = __fmaf_rn(0.5f, fabsf(d), __fadd_rn(fabsf(bhc), fabsf(b3c)));
    // |fl(Delta) - Delta| <= u (78 Q^2 mQ + 12 |Q|^3 + 88 |R| mR + 4 R^2) with u = 2^-24
    // (a factor 2 over the first-order propagation of the roundings above,
    // with a reciprocal of A off by up to 2 ulp).  As |Q|^3 <= Q^2 mQ and
    // R^2 <= |R| mR, that is at most 92 u (Q^2 mQ + |R| mR); the bound takes
    // 128 u (Q^2 mQ + |R| mR), a safety factor of 1.39.
    const float bound = __fmul_rn(7.68e-6f, __fmaf_rn(Qs, mQ, __fmul_rn(fabsf(R), mR)));
    int branch; // 0 Cardano, 1 triple, 2 trig
    if (Dl > bound) branch = 0;
    else if (Dl < -bound) branch = 2;
    else { // among them every A whose reciprocal left the range: Delta is 0 or NaN, or the bound infinite
        ++esc;
        if (!rcp_in_range(inv)) return quartic_min_fallback64(A, B, C, D, lo, hi, paper_mode);
        branch = cubic_branch64(A, B, C, D);
    }
    if (branch == 1) return clampf(-b3, lo, hi);
    if (branch == 0) {
        // Delta > 0 here (certified, or FP64 said so)
        const float sq = Dl > 0.0f ? __fmul_rn(Dl, rsqrt_fast(Dl)) : 0.0f;
        const float S = cbrt_fast(__fadd_rn(R, R >= 0.0f ? sq : -sq));
        const float T = S != 0.0f ? __fmul_rn(-Q, rcp_fast(S)) : 0.0f;
        const float x = newton_polish32(A, B, C, D, __fsub_rn(__fadd_rn(S, T), b3));
        if (!isfinite(x)) return quartic_min_fallback64(A, B, C, D, lo, hi, paper_mode);
        return clampf(x, lo, hi);
    }
    // three real roots: t = theta/3 lies in [0, pi/3], where the fast sine and
    // cosine are accurate to a few ulp; the Newton step below removes their error
    const float nQ = fmaxf(-Q, 0.0f);
    const float arg = nQ > 0.0f ? fminf(fmaxf(R * rsqrtf(nQ * nQ * nQ), -1.0f), 1.0f) : (R >= 0.0f ? 1.0f : -1.0f);
    const float t = acosf(arg) * (1.0f / 3.0f);
    const float st = __sinf(t), ct = __cosf(t);
    const float two_sq = 2.0f * sqrt_fast(nQ);
    float x3 = two_sq * ct - b3;
    float x1 = two_sq * (-0.5f * ct - 0.86602540378f * st) - b3;
    x1 = newton_polish32(A, B, C, D, x1);
    x3 = newton_polish32(A, B, C, D, x3);
    if (!isfinite(x1) || !isfinite(x3)) return quartic_min_fallback64(A, B, C, D, lo, hi, paper_mode);
    if (paper_mode) {
        const float xs = delta_f32(x1, x3, b, c, d) > 0.0f ? x3 : x1;
        return clampf(xs, lo, hi);
    }
    const float u = clampf(x1, lo, hi), v = clampf(x3, lo, hi);
    return delta_f32(u, v, b, c, d) > 0.0f ? v : u;
}

// cos(acos(a) / 3) for a in [-1, 1], whose 2 sqrt(-Q)-fold is the largest
// root of z^3 + 3 Q z - 2 R with a = R / sqrt(-Q)^3 (and, of -a, minus the
// smallest): with w = sqrt((1 + a) / 2) = cos(acos(a) / 2) it is
// cos((2/3) acos w), analytic on [0, 1] (the nearest singularity is w = -1), here
// by its degree-7 Chebyshev interpolant (error 1e-7 in FP32 arithmetic).
__device__ __forceinline__ float sqrt_approx(float v)
{
    float r;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(v));
    return r;
}
#define ADMM_THIRD_COEFS                                                                                   \
    {0.5f, 0.577347219f, -0.111043237f, 0.0528691076f, -0.0303130634f, 0.0161594898f, -0.00616994966f, 0.00115042902f}
__device__ __forceinline__ float cos_third(float a)
{
    const float k[8] = ADMM_THIRD_COEFS;
    const float w = sqrt_approx(fmaf(0.5f, a, 0.5f));
    float r = k[7];
#pragma unroll
    for (int t = 6; t >= 0; --t) r = fmaf(r, w, k[t]);
    return r;
}

// Newton step and slope of the derivative's half H(x) = 2A x^3 + 1.5B x^2 + C x + D/2 in FP32.
__device__ __forceinline__ void half_polish32(float A2, float B15, float C, float Dh, float &x, float &s)
{
    const float h = fmaf(fmaf(fmaf(A2, x, B15), x, C), x, Dh);
    const float sl = fmaf(fmaf(3.0f * A2, x, 2.0f * B15), x, C);
    const float dx = h * rcp_fast(sl);
    if (sl > 0.0f && fabsf(dx) <= 0.0625f * (fabsf(x) + 1.0f)) x -= dx;
    s = fmaf(fmaf(3.0f * A2, x, 2.0f * B15), x, C);
}

// ---------------------------------------------------------------------------
// FP64 minimiser seeded in FP32.  FP64 throughput is 1/64 of FP32 on this
// GPU, so everything that can be decided in FP32 with certainty is: the
// branch of the cubic (the error bound of quartic_min32, doubled for the
// rounding of A, B, C, D to FP32), and on the trig branch which of the two
// minima is the constrained minimiser (the sign of F(u) - F(v) = (u - v) br
// where |br| exceeds 1e-5 of the sum of its terms' magnitudes; FP32 makes an
// error of a few 1e-7 of it).  Only the chosen root is refined, by two FP64
// Newton steps on half the derivative with one FP32 slope: 9 FP64-pipe
// instructions in all, where both closed forms took 186 per warp.  Anything
// uncertain, out of the FP32 range, or not settled takes the FP64 closed form.
// 1e6 quartics (a third of them double wells): 571 -> 43 us a call on device arrays (kernel 381 -> 29 us).
// ---------------------------------------------------------------------------
static __device__ __noinline__ double quartic_min64_closed(double A, double B, double C, double D, double lo,
                                                           double hi, int paper_mode)
{
    return quartic_min64(A, B, C, D, lo, hi, paper_mode);
}

// FP32 root to refine (x) and the slope of H there (s); false: not certain.
__device__ __forceinline__ bool quartic_seed32(float A, float B, float C, float D, float lo, float hi,
                                               int paper_mode, float &x, float &s)
{
    const float inv = rcp_fast(A);
    const float b = 0.75f * B * inv, c = 0.5f * C * inv, d = 0.25f * D * inv;
    const float b3 = b * (1.0f / 3.0f);
    const float Q = c * (1.0f / 3.0f) - b3 * b3;
    const float R = b3 * (0.5f * c) - b3 * b3 * b3 - 0.5f * d;
    const float Q3 = Q * Q * Q, R2 = R * R;
    const float Dl = Q3 + R2;
    const float mQ = fabsf(c) * (1.0f / 3.0f) + b3 * b3;
    const float mR = fabsf(b3 * 0.5f * c) + fabsf(b3 * b3 * b3) + 0.5f * fabsf(d);
    const float bound = 1.2e-7f * (96.0f * Q * Q * mQ + 64.0f * fabsf(Q3) + 96.0f * fabsf(R) * mR + 64.0f * R2);
    const float A2 = A + A, B15 = 1.5f * B, Dh = 0.5f * D;
    if (Dl > bound) {
        const float sq = sqrt_fast(Dl);
        const float S = cbrt_fast(R >= 0.0f ? R + sq : R - sq);
        x = S - Q * rcp_fast(S) - b3;
        half_polish32(A2, B15, C, Dh, x, s);
        return true;
    }
    if (!(Dl < -bound)) return false;
    const float rs = rsqrt_fast(-Q), sq2 = 2.0f * -Q * rs;
    const float arg = fminf(fmaxf(R * (rs * rs * rs), -1.0f), 1.0f);
    float x3 = fmaf(sq2, cos_third(arg), -b3), x1 = fmaf(-sq2, cos_third(-arg), -b3), s1, s3;
    half_polish32(A2, B15, C, Dh, x1, s1);
    half_polish32(A2, B15, C, Dh, x3, s3);
    float u = x1, v = x3;
    bool third = false;
    if (!paper_mode) {
        u = clampf(x1, lo, hi);
        v = clampf(x3, lo, hi);
        // both minima on one side of the interval: the same end of it
        if (x3 < lo - 1.0e-5f * (fabsf(lo) + 1.0f) || x1 > hi + 1.0e-5f * (fabsf(hi) + 1.0f)) u = v;
        else if (!(v - u > 1.0e-4f * (fabsf(u) + fabsf(v) + 1.0f))) return false;
    }
    if (u != v) {
        const float uu = u * u, vv = v * v, uv = u * v;
        const float t3 = A * (u + v) * (uu + vv), t2 = B * (uu + uv + vv), t1 = C * (u + v); // u^3 + u^2 v + u v^2 + v^3
        const float m3 = A * (fabsf(u) + fabsf(v)) * (uu + vv), m2 = fabsf(B) * (uu + fabsf(uv) + vv),
                    m1 = fabsf(C) * (fabsf(u) + fabsf(v));
        const float br = t3 + t2 + t1 + D;
        if (!(fabsf(br) > 1.0e-5f * (m3 + m2 + m1 + fabsf(D)))) return false;
        third = br < 0.0f; // u < v: F(u) > F(v)
    }
    x = third ? x3 : x1;
    s = third ? s3 : s1;
    return true;
}

// v / 2 on the integer pipes (a denormal result gives a signed zero)
__device__ __forceinline__ double half64(double v)
{
    const int h = __double2hiint(v);
    const bool z = (h & 0x7ff00000) <= 0x00100000;
    return __hiloint2double(z ? h & 0x80000000 : h - 0x00100000, z ? 0 : __double2loint(v));
}

__device__ __forceinline__ bool newton_settled(float d0, float d1, float x);

// Called by whole warps: the lanes come together again before the FP64
// refinement, which a warp with several branches would otherwise run once for each
// (30 FP64 instructions per warp instead of 10).
__device__ __forceinline__ double quartic_min64_seeded(double A, double B, double C, double D, double lo, double hi,
                                                       int paper_mode)
{
    const bool lin = (__double_as_longlong(A) << 1) == 0; // A = 0: B plays no part
    const float Af = f64_to_f32_int(A), Cf = f64_to_f32_int(C), Df = f64_to_f32_int(D);
    float xf = 0.0f, sf = 0.0f;
    if (lin) {
        xf = -0.5f * Df * rcp_fast(Cf);
        sf = Cf;
    } else if (Af > 1.0e-30f && Af < 1.0e30f) {
        if (!quartic_seed32(Af, f64_to_f32_int(B), Cf, Df, f64_to_f32_int(lo), f64_to_f32_int(hi), paper_mode, xf, sf))
            sf = 0.0f;
    }
    __syncwarp();
    const float rf = rcp_fast(sf);
    // A lies in the FP32 range, so doubling it is one more in the exponent
    const double A2 = lin ? 0.0 : __longlong_as_double(__double_as_longlong(A) + 0x0010000000000000ll);
    const double B15 = lin ? 0.0 : 1.5 * B, Dh = half64(D), r = f32_to_f64_int(rf);
    double x = f32_to_f64_int(xf);
    float dn[2];
#pragma unroll
    for (int t = 0; t < 2; ++t) {
        const double H = fma(fma(fma(A2, x, B15), x, C), x, Dh);
        x = fma(-H, r, x);
        dn[t] = f64_to_f32_int(H) * rf;
    }
    if (sf > 0.0f && isfinite(xf) && isfinite(rf) && rf >= 1.2e-38f && newton_settled(dn[0], dn[1], xf))
        return clamp_ord(x, lo, hi);
    return quartic_min64_closed(A, B, C, D, lo, hi, paper_mode);
}

// ---------------------------------------------------------------------------
// Step (a) of one element in FP64, in the factored form of its terms of L:
//   (a_2/q + rho_3/2) x^2 + (a_1/q - rho_3 phi) x + (rho_1/2) (b_2 x^2 + b_1 x - u)^2
// (plus the rho_4 terms at k = 0).  Half its derivative is
//   H(x) = C x + Dh + hr1 e g',  e = b_2 x^2 + b_1 x - u,  g' = 2 b_2 x + b_1,  hr1 = rho_1/2,
// six FP64 instructions, against twelve to expand A, B, C, D and three per
// Horner evaluation.  The root is found in FP32 (closed form of the cubic in
// z = x + b_1/(2 b_2), where it is already depressed, then a Newton step on H)
// and refined by two FP64 Newton steps with one FP32 slope: each multiplies
// the error by the slope's relative error.  21 FP64-pipe instructions per
// element with losses and 7 without, where expanding the quartic and
// converting and comparing on the FP64 pipe took about 80 and 25.
// ---------------------------------------------------------------------------
struct Elem64 {
    double b2, b1, u, C, Dh, hr1;
};

// The FP64 closed form of Algorithm 1, out of line: the trig and triple-root
// branches, a discriminant FP32 cannot certify, values outside the FP32 range, a
// Newton step that did not settle.
static __device__ __noinline__ double elem_min64(Elem64 p, double lo, double hi, int paper_mode)
{
    const double A = p.hr1 * p.b2 * p.b2, B = 2.0 * p.hr1 * p.b2 * p.b1;
    const double C = p.C + p.hr1 * (p.b1 * p.b1 - 2.0 * p.b2 * p.u), D = 2.0 * (p.Dh - p.hr1 * p.b1 * p.u);
    return quartic_min64(A, B, C, D, lo, hi, paper_mode);
}

// One Newton step on H in FP32, then 1 / H' at the new point; false where H'
// is not positive there or a value left the FP32 range.
__device__ __forceinline__ bool elem_polish32(float b2, float b1, float u, float C, float Dh, float hr1, float y,
                                              float &x, float &r)
{
    const float t = fmaf(b2, y, b1), e = fmaf(t, y, -u), gp = fmaf(b2, y, t);
    const float dx = fmaf(e * gp, hr1, fmaf(C, y, Dh)) * rcp_fast(fmaf(hr1, fmaf(gp, gp, 2.0f * b2 * e), C));
    if (fabsf(dx) <= 0.0625f * (fabsf(y) + 1.0f)) y -= dx;
    const float t1 = fmaf(b2, y, b1), e1 = fmaf(t1, y, -u), gp1 = fmaf(b2, y, t1);
    const float s = fmaf(hr1, fmaf(gp1, gp1, 2.0f * b2 * e1), C);
    x = y;
    r = rcp_fast(s);
    return fabsf(x) < 1.0e30f && r >= 1.2e-38f && r < 1.0e38f;
}

// The minimiser's FP32 root where H has three real roots (Delta < 0
// certified, Q < 0): with z = x + b_1/(2 b_2) the quartic is z^4/4 + (3/2) Q z^2
// - 2 R z up to scale, so
//  * where [lo, hi] lies right of z = sqrt(-Q) (left of -sqrt(-Q)), H
//    increases on it and the constrained minimiser is the clamped largest
//    (smallest) root;
//  * the lower of the two minima is the one on the side of R's sign; it is
//    the constrained minimiser too if it lies inside (lo, hi).
// Anything else (a minimum outside the interval that holds the other) is left
// to the FP64 closed form.  dR bounds R's error.  Out of line: rare.
static __device__ __noinline__ bool elem_trig32(float Q, float R, float dR, float b3, float lo, float hi,
                                                int paper_mode, float &y)
{
    const float nQ = -Q, s = sqrt_fast(nQ); // nQ > 0: Delta < 0 is certified
    const float mlo = 1.0e-5f * (fabsf(lo) + fabsf(b3) + 1.0f), mhi = 1.0e-5f * (fabsf(hi) + fabsf(b3) + 1.0f);
    int side = 0;
    if (!paper_mode) {
        if (lo + b3 - mlo > 1.0001f * s) side = 1;
        else if (hi + b3 + mhi < -1.0001f * s) side = -1;
    }
    const bool basin = side != 0;
    if (!basin) {
        if (!(fabsf(R) > dR)) return false;
        side = R > 0.0f ? 1 : -1;
    }
    const float Rs = side > 0 ? R : -R;
    const float rs = rsqrt_fast(nQ);
    const float arg = fminf(fmaxf(Rs * (rs * rs * rs), -1.0f), 1.0f);
    const float z = 2.0f * s * __cosf(acosf(arg) * (1.0f / 3.0f));
    y = (side > 0 ? z : -z) - b3;
    return basin || paper_mode || (y > lo + mlo && y < hi - mhi);
}

// FP32 root of H (x) and 1 / H'(x) (r) that the minimiser is refined from:
// the quadratic case (b_2 = 0), the Cardano branch with Delta > 0 certified,
// and the trig branch with Delta < 0 certified where elem_trig32 can tell the root.
// Q and R carry the truncation of b_2, b_1, u, C, Dh to FP32 (2 v, v = 2^-24),
// the rounding of their own operations and two reciprocals off by 2 ulp: |dQ|
// <= 30 v mQ, |dR| <= 22 v mR (mQ, mR the sums of the terms' magnitudes), so
// |dDelta| <= v (94 Q^2 mQ + 48 |R| mR); the bound takes 128 v for both.
__device__ __forceinline__ bool elem_seed32(float b2, float b1, float u, float C, float Dh, float hr1, double lo,
                                            double hi, int paper_mode, float &x, float &r)
{
    if (!(fabsf(b1) + fabsf(u) + C + fabsf(Dh) < 1.0e37f)) return false; // cut off at the end of the FP32 range
    if (b2 <= 1.2e-38f) { // 0 (or below the FP32 range): the converted value is the smallest normal one
        const float hb1 = hr1 * b1;
        r = rcp_fast(fmaf(hb1, b1, C));
        x = fmaf(hb1, u, -Dh) * r;
        return fabsf(x) < 1.0e30f && r >= 1.2e-38f && r < 1.0e38f;
    }
    const float b3 = 0.5f * b1 * rcp_fast(b2);
    const float v = 0.5f * b1 * b3;                 // b_1^2 / (4 b_2)
    const float k2 = (hr1 + hr1) * b2;
    const float inv = rcp_fast(k2 * b2), inv3 = inv * (1.0f / 3.0f), inv2 = 0.5f * inv;
    const float Q = (C - k2 * (u + v)) * inv3, R = (C * b3 - Dh) * inv2;
    const float mQ = (C + k2 * (fabsf(u) + fabsf(v))) * inv3, mR = (C * fabsf(b3) + fabsf(Dh)) * inv2;
    const float Qs = Q * Q;
    const float Dl = fmaf(Qs, Q, R * R);
    const float bound = 7.68e-6f * fmaf(Qs, mQ, fabsf(R) * mR);
    float y;
    if (Dl > bound) {
        const float sq = sqrt_fast(Dl);
        const float S = cbrt_fast(R >= 0.0f ? R + sq : R - sq);
        y = S - Q * rcp_fast(S) - b3;
    } else if (!(Dl < -bound) || !elem_trig32(Q, R, 2.0e-6f * mR, b3, f64_to_f32_seed(lo), f64_to_f32_seed(hi), paper_mode, y)) {
        return false;
    }
    return elem_polish32(b2, b1, u, C, Dh, hr1, y, x, r);
}

// The settled test of two Newton steps d0, d1 of a refined root: the second
// step's own error is d1 times the ratio of the steps.
__device__ __forceinline__ bool newton_settled(float d0, float d1, float x)
{
    const float s = fabsf(x) + 1.0f, a = fabsf(d1);
    return a <= 1.0e-12f * s || (a <= 1.0e-10f * s && a <= 1.0e-5f * fabsf(d0));
}

// A certified root whose FP32 seed was too far off for two steps (a tiny b_2:
// x is a small difference of numbers of size b_1 / b_2): Newton steps with FP64
// slopes, which keep FP64's precision where the closed form loses it to that
// difference (3.8e-10 at b_2 = 1e-6, b_1 = 1).  False: not settled either.
static __device__ __noinline__ bool elem_refine64(Elem64 p, double &x)
{
    double y = x, last = INFINITY;
    for (int t = 0; t < 8; ++t) {
        const double w = fma(p.b2, y, p.b1), e = fma(w, y, -p.u), gp = fma(p.b2, y, w);
        const double s = fma(p.hr1, fma(gp, gp, 2.0 * p.b2 * e), p.C);
        if (!(s > 0.0)) return false;
        const double d = fma(e * gp, p.hr1, fma(p.C, y, p.Dh)) / s;
        y -= d;
        if (fabs(d) <= 1.0e-15 * (fabs(y) + 1.0)) return x = y, true;
        if (t > 3 && !(fabs(d) < 0.5 * last)) return false;
        last = fabs(d);
    }
    return false;
}

// The constrained minimiser of an element with losses (b_2 or b_1 not zero).
__device__ __forceinline__ double elem_min64_seeded(const Elem64 &p, float hr1f, double lo, double hi, int paper_mode)
{
    float xf, rf;
    if (elem_seed32(f64_to_f32_seed(p.b2), f64_to_f32_seed(p.b1), f64_to_f32_seed(p.u), f64_to_f32_seed(p.C),
                    f64_to_f32_seed(p.Dh), hr1f, lo, hi, paper_mode, xf, rf)) {
        const double r = f32_to_f64_seed(rf);
        double x = f32_to_f64_seed(xf);
        float d[2];
#pragma unroll
        for (int t = 0; t < 2; ++t) {
            const double w = fma(p.b2, x, p.b1), e = fma(w, x, -p.u), gp = fma(p.b2, x, w);
            const double H = fma(e * gp, p.hr1, fma(p.C, x, p.Dh));
            x = fma(-H, r, x);
            d[t] = f64_to_f32_seed(H) * rf;
        }
        if (newton_settled(d[0], d[1], xf) || elem_refine64(p, x)) return clamp_ord(x, lo, hi);
    }
    return elem_min64(p, lo, hi, paper_mode);
}

// The same without losses: H(x) = C x + Dh.  A Dh beyond the FP32 range (an
// infinity or a NaN too, which the seed's conversion makes finite) takes the
// division and the comparing clamp.
__device__ __forceinline__ double elem_min64_linear(double C, double Dh, double lo, double hi)
{
    const float Cf = f64_to_f32_seed(C), Df = f64_to_f32_seed(Dh), rf = rcp_fast(Cf), xf = -Df * rf;
    if (rf >= 1.2e-38f && rf < 1.0e38f && fabsf(xf) < 1.0e30f && fabsf(Df) < 1.0e37f) {
        const double r = f32_to_f64_seed(rf);
        double x = f32_to_f64_seed(xf);
        x = fma(-fma(C, x, Dh), r, x);
        x = fma(-fma(C, x, Dh), r, x);
        return clamp_ord(x, lo, hi);
    }
    return clampd(-Dh / C, lo, hi);
}

// ---------------------------------------------------------------------------
// Packed pair variant: the two columns of a vector in one float2, on the
// paired FP32 instructions (FADD2 / FMUL2 / FFMA2: two lanes per issue, the
// same rounding per lane as the scalar operations).  The common cases run
// packed: both lanes quadratic (A = 0), or both lanes on the Cardano branch
// with the discriminant's sign certified.  Any other combination (trig or
// uncertain branch, mixed A = 0 / A > 0, non-finite intermediate) is solved
// lane by lane by quartic_min32, so each lane gets the branch Algorithm 1
// gives it.
// ---------------------------------------------------------------------------
// Written as PTX, each with its own rounding: the compiler fuses the builtins'
// products into later sums where a product has one use, which made the bits
// depend on what else a copy of the code needed the product for.
__device__ __forceinline__ float2 add2(float2 a, float2 b)
{
    float2 r;
    asm("{.reg .b64 p, q, s; mov.b64 p, {%2, %3}; mov.b64 q, {%4, %5}; add.rn.f32x2 s, p, q; mov.b64 {%0, %1}, s;}"
        : "=f"(r.x), "=f"(r.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return r;
}
__device__ __forceinline__ float2 mul2(float2 a, float2 b)
{
    float2 r;
    asm("{.reg .b64 p, q, s; mov.b64 p, {%2, %3}; mov.b64 q, {%4, %5}; mul.rn.f32x2 s, p, q; mov.b64 {%0, %1}, s;}"
        : "=f"(r.x), "=f"(r.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return r;
}
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c)
{
    float2 r;
    asm("{.reg .b64 p, q, s, t; mov.b64 p, {%2, %3}; mov.b64 q, {%4, %5}; mov.b64 t, {%6, %7};"
        " fma.rn.f32x2 s, p, q, t; mov.b64 {%0, %1}, s;}"
        : "=f"(r.x), "=f"(r.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
    return r;
}
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return fma2(b, make_float2(-1.0f, -1.0f), a); }
__device__ __forceinline__ float2 splat2(float v) { return make_float2(v, v); }
__device__ __forceinline__ float2 neg2(float2 a) { return mul2(a, make_float2(-1.0f, -1.0f)); }
__device__ __forceinline__ float2 abs2(float2 a) { return make_float2(fabsf(a.x), fabsf(a.y)); }

// Newton step of newton_polish32 on both lanes.
__device__ __forceinline__ float2 newton_polish32x2(float2 A, float2 B, float2 C, float2 D, float2 x)
{
    const float2 A4 = mul2(splat2(4.0f), A), B3 = mul2(splat2(3.0f), B), C2 = add2(C, C);
    const float2 fp = fma2(fma2(fma2(A4, x, B3), x, C2), x, D);
    const float2 fpp = fma2(fma2(mul2(splat2(12.0f), A), x, mul2(splat2(6.0f), B)), x, C2);
    const float2 r = make_float2(rcp_fast(fpp.x), rcp_fast(fpp.y)); // used only where fpp > 0
    const float2 dx = mul2(fp, r);
    const float2 xn = sub2(x, dx);
    const float2 lim = mul2(splat2(0.0625f), add2(abs2(x), splat2(1.0f)));
    return make_float2((fpp.x > 0.0f && fabsf(dx.x) <= lim.x) ? xn.x : x.x,
                       (fpp.y > 0.0f && fabsf(dx.y) <= lim.y) ? xn.y : x.y);
}

// Lane by lane (out of line: the rare path stays out of the element loop).
static __device__ __noinline__ float2 quartic_min32_lanes(float2 A, float2 B, float2 C, float2 D, float2 lo,
                                                          float2 hi, int paper_mode, unsigned *esc)
{
    unsigned e = *esc;
    const float2 x = make_float2(quartic_min32(A.x, B.x, C.x, D.x, lo.x, hi.x, paper_mode, e),
                                 quartic_min32(A.y, B.y, C.y, D.y, lo.y, hi.y, paper_mode, e));
    *esc = e;
    return x;
}

// In step (a) 2 C is at least rho_3 where A = 0, so a test of rho_3 says whether it may be denormal.
__device__ __forceinline__ bool tiny_rho3(float rho3) { return rho3 < 1.17549435e-38f; }

// tiny_c: 2 C may be denormal where A = 0, so look for an infinite reciprocal.
__device__ __forceinline__ float2 quartic_min32x2(float2 A, float2 B, float2 C, float2 D, float2 lo, float2 hi,
                                                  int paper_mode, unsigned &esc, bool tiny_c)
{
#ifndef ADMM_COMPENSATED_POLISH
    if (A.x > 0.0f && A.y > 0.0f) {
        const float2 inv = make_float2(rcp_fast(A.x), rcp_fast(A.y));
        const float2 b = mul2(mul2(splat2(0.75f), B), inv);
        const float2 c = mul2(mul2(splat2(0.5f), C), inv);
        const float2 d = mul2(mul2(splat2(0.25f), D), inv);
        const float2 b3 = mul2(b, splat2(1.0f / 3.0f));
        const float2 b3s = mul2(b3, b3);
        const float2 nQ = fma2(c, splat2(-1.0f / 3.0f), b3s); // -Q
        const float2 hc = mul2(splat2(0.5f), c), nhd = mul2(splat2(-0.5f), d);
        const float2 R = fma2(b3, sub2(hc, b3s), nhd);
        const float2 Qs = mul2(nQ, nQ);
        const float2 Dl = fma2(neg2(Qs), nQ, mul2(R, R));
        // the forward error bound of quartic_min32, on both lanes
        const float2 mQ = fma2(abs2(c), splat2(1.0f / 3.0f), b3s);
        const float2 mR = fma2(abs2(b3), add2(b3s, abs2(hc)), abs2(nhd));
        const float2 bound = mul2(splat2(7.68e-6f), fma2(Qs, mQ, mul2(abs2(R), mR)));
        if (Dl.x > bound.x && Dl.y > bound.y) { // Cardano on both lanes
            // here Delta > bound >= 0, so sqrt(Delta) > 0, |R +- sqrt(Delta)| > 0 and S != 0: the
            // zero guards of sqrt_fast, cbrt_fast and the T reciprocal are not needed (an S that
            // underflows gives a non-finite x and the lane-by-lane path below)
            const float2 sq = mul2(Dl, make_float2(rsqrt_fast(Dl.x), rsqrt_fast(Dl.y)));
            const float2 v = add2(R, make_float2(R.x >= 0.0f ? sq.x : -sq.x, R.y >= 0.0f ? sq.y : -sq.y));
            const float2 S = make_float2(copysignf(cbrt_abs(v.x), v.x), copysignf(cbrt_abs(v.y), v.y));
            const float2 rS = make_float2(rcp_fast(S.x), rcp_fast(S.y));
            const float2 x = newton_polish32x2(A, B, C, D, sub2(fma2(nQ, rS, S), b3)); // S + T - b/3
            if (isfinite(x.x) && isfinite(x.y))
                return make_float2(clampf(x.x, lo.x, hi.x), clampf(x.y, lo.y, hi.y));
        }
    }
    if (A.x == 0.0f && A.y == 0.0f) { // quadratic on both lanes
        const float2 C2 = add2(C, C);
        const float2 r = make_float2(rcp_fast(C2.x), rcp_fast(C2.y)), x = mul2(neg2(D), r);
        if (!tiny_c || r.x * r.y < INFINITY) // (two finite ones whose product is not: the same bits lane by lane)
            return make_float2(clampf(x.x, lo.x, hi.x), clampf(x.y, lo.y, hi.y));
    }
#endif
    return quartic_min32_lanes(A, B, C, D, lo, hi, paper_mode, &esc);
}

// The same for many quartics with any mix of single and double wells (the
// quartic benchmark, where a third are double wells and nearly every warp holds
// both branches): both lanes' Cardano root and both lanes' trig roots are found
// packed, and each lane keeps what its branch needs, instead of one lane after
// the other through the scalar code (725 -> 284 warp instructions per 64
// quartics, 2^26 of them 1014 -> 350 us).  The decisions are those of quartic_min32: the branch outside
// its error bound, the lower minimum where |br| of F(u) - F(v) = (u - v) br
// exceeds 2e-5 of the sum of its terms' magnitudes (FP32 errs by a few 1e-7
// of it).  okx, oky: a lane with anything nearer than that, A = 0, or a value that
// is not finite is left to quartic_min32.  Each lane's result depends on its own
// element alone.
__device__ __forceinline__ float2 min2(float2 a, float2 b) { return make_float2(fminf(a.x, b.x), fminf(a.y, b.y)); }
__device__ __forceinline__ float2 max2(float2 a, float2 b) { return make_float2(fmaxf(a.x, b.x), fmaxf(a.y, b.y)); }
__device__ __forceinline__ float2 sel2(bool px, bool py, float2 a, float2 b)
{
    return make_float2(px ? a.x : b.x, py ? a.y : b.y);
}
__device__ __forceinline__ float2 cos_third2(float2 a)
{
    const float2 h = fma2(splat2(0.5f), a, splat2(0.5f));
    const float2 w = make_float2(sqrt_approx(h.x), sqrt_approx(h.y));
    const float k[8] = ADMM_THIRD_COEFS;
    float2 r = splat2(k[7]);
#pragma unroll
    for (int t = 6; t >= 0; --t) r = fma2(r, w, splat2(k[t]));
    return r;
}

__device__ __forceinline__ float2 quartic_min32x2_wells(float2 A, float2 B, float2 C, float2 D, float2 lo, float2 hi,
                                                        int paper_mode, bool &okx, bool &oky)
{
    const float2 inv = make_float2(rcp_fast(A.x), rcp_fast(A.y));
    const float2 b = mul2(mul2(splat2(0.75f), B), inv);
    const float2 c = mul2(mul2(splat2(0.5f), C), inv);
    const float2 d = mul2(mul2(splat2(0.25f), D), inv);
    const float2 b3 = mul2(b, splat2(1.0f / 3.0f));
    const float2 b3s = mul2(b3, b3);
    const float2 nQ = fma2(c, splat2(-1.0f / 3.0f), b3s); // -Q
    const float2 hc = mul2(splat2(0.5f), c), nhd = mul2(splat2(-0.5f), d);
    const float2 R = fma2(b3, sub2(hc, b3s), nhd);
    const float2 Qs = mul2(nQ, nQ);
    const float2 Dl = fma2(neg2(Qs), nQ, mul2(R, R));
    // the forward error bound of quartic_min32, on both lanes
    const float2 ahc = abs2(hc), ahd = abs2(nhd), nb3 = neg2(b3);
    const float2 mQ = fma2(ahc, splat2(2.0f / 3.0f), b3s);
    const float2 mR = fma2(abs2(b3), add2(b3s, ahc), ahd);
    const float2 bound = mul2(splat2(7.68e-6f), fma2(Qs, mQ, mul2(abs2(R), mR)));
    const bool cx = Dl.x > bound.x, cy = Dl.y > bound.y, tx = Dl.x < -bound.x, ty = Dl.y < -bound.y;
    okx = A.x > 0.0f && (cx || tx);
    oky = A.y > 0.0f && (cy || ty);
    // sqrt(Delta) on the Cardano branch, sqrt(-Q) on the trig branch
    const float2 rad = sel2(cx, cy, Dl, nQ);
    const float2 rs = make_float2(rsqrt_fast(rad.x), rsqrt_fast(rad.y));
    const float2 sq = mul2(rad, rs);
    float2 u, v = splat2(0.0f); // Cardano: the root; trig: the smallest and the largest root
    {
        const float2 w = add2(R, make_float2(R.x >= 0.0f ? sq.x : -sq.x, R.y >= 0.0f ? sq.y : -sq.y));
        const float2 S = make_float2(copysignf(cbrt_abs(w.x), w.x), copysignf(cbrt_abs(w.y), w.y));
        u = add2(fma2(nQ, make_float2(rcp_fast(S.x), rcp_fast(S.y)), S), nb3);
    }
    const bool any_trig = __any_sync(__activemask(), tx || ty);
    if (any_trig) {
        const float2 arg = max2(min2(mul2(R, mul2(rs, mul2(rs, rs))), splat2(1.0f)), splat2(-1.0f));
        const float2 sq2 = add2(sq, sq);
        v = fma2(sq2, cos_third2(arg), nb3);
        u = sel2(tx, ty, fma2(neg2(sq2), cos_third2(neg2(arg)), nb3), u);
        v = newton_polish32x2(A, B, C, D, v);
        v = sel2(tx, ty, v, u);
    }
    u = newton_polish32x2(A, B, C, D, u);
    const float2 fin = fma2(u, splat2(0.0f), mul2(v, splat2(0.0f))); // 0 where u and v are finite, else NaN
    okx = okx && fin.x == 0.0f;
    oky = oky && fin.y == 0.0f;
    float2 x = max2(min2(u, hi), lo);
    if (any_trig) {
        const float2 vc = max2(min2(v, hi), lo);
        const float2 p = paper_mode ? u : x, r = paper_mode ? v : vc;
        const float2 s = add2(p, r), q2 = fma2(p, p, mul2(r, r)), q3 = fma2(p, r, q2);
        const float2 as = add2(abs2(p), abs2(r)), b3q = mul2(b3, q3);
        // br = (u^3 + u^2 v + u v^2 + v^3) / 4 + (b/3) (u^2 + u v + v^2) + (c/2) (u + v) + d
        const float2 q4 = mul2(splat2(0.25f), q2);
        const float2 br = add2(fma2(q4, s, b3q), fma2(hc, s, d));
        const float2 mb = add2(fma2(q4, as, abs2(b3q)), fma2(ahc, as, add2(ahd, ahd)));
        const float2 lim = mul2(splat2(2.0e-5f), mb);
        const bool nx = tx && p.x != r.x, ny = ty && p.y != r.y; // u < v: the larger root where br < 0
        okx = okx && (!nx || fabsf(br.x) > lim.x);
        oky = oky && (!ny || fabsf(br.y) > lim.y);
        x = sel2(nx && br.x < 0.0f, ny && br.y < 0.0f, vc, x);
    }
    return x;
}

} // namespace admm_impl
