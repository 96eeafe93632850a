// lf2_arith.cuh -- the device arithmetic every leapfrog kernel of liblf2 compiles: coefficient
// packs, the per-site update functions and the lattice geometry helpers.
//
// Every kernel variant (one thread per site, z-streaming tiles, temporal blocking, ensemble)
// performs the per-site update through the functions below, written with explicit
// round-to-nearest intrinsics so that the compiler cannot contract or reorder them
// differently in different kernels: all variants give bitwise identical results (but for the sign of
// an exact zero in temporal blocking on packed pairs, see lf2_tblock.cuh).
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

#include "../../include/lf2.h"

namespace lf2 {

constexpr int kMaxComp = LF2_MAX_COMP;

// ---------------------------------------------------------------- coefficient packs
// FP64: the force enters only through dt*F, folded as
//   dt F_a = a * nb_a - (dl * s2 + b0) * phi_a
// with nb_a the sum of the 6 neighbours, s2 = sum_b phi_b^2 and
//   a = dt/dx^2,  dl = dt lambda,  b0 = dt (6/dx^2 + m2 - lambda eta^2).
struct Coef64 {
    double a, dl, b0, dt;
};

// FP32: difference form of the Laplacian (sum_i (phi(x+-i) - phi(x))), which keeps the
// small differences of a smooth field exact when |phi| ~ eta, then
//   F_a = d_a * inv_dx2 - (lambda (s2 - eta^2) + m2) phi_a.
struct Coef32 {
    float inv_dx2, lam, eta2, m2, dt;
    float zero;  // always 0: a run-time zero for the packed path (see make_coef32x2)
};

// Energy (always FP64).  The synchronised momentum pi_n = pi_{n-1/2} + (dt/2) F(phi_n) is a
// kick of half a step, folded as in Coef64 with dt/2: ah = (dt/2)/dx^2, hl = (dt/2) lambda,
// hb0 = (dt/2)(6/dx^2 + m2 - lambda eta^2).  The remaining members scale the raw sums.
struct CoefE {
    double ah, hl, hb0, eta2;
    double inv_dx2, lam, m2, vol;  // vol = dx^3
};

inline Coef64 make_coef64(const lf2_params &p, double dt) {
    const double inv_dx2 = 1.0 / (p.dx * p.dx);
    return Coef64{dt * inv_dx2, dt * p.lambda, dt * (6.0 * inv_dx2 + p.m2 - p.lambda * p.eta * p.eta), dt};
}

inline Coef32 make_coef32(const lf2_params &p, double dt) {
    return Coef32{(float)(1.0 / (p.dx * p.dx)), (float)p.lambda, (float)(p.eta * p.eta), (float)p.m2, (float)dt, 0.0f};
}

inline CoefE make_coefE(const lf2_params &p) {
    const double inv_dx2 = 1.0 / (p.dx * p.dx), h = 0.5 * p.dt;
    return CoefE{h * inv_dx2, h * p.lambda, h * (6.0 * inv_dx2 + p.m2 - p.lambda * p.eta * p.eta), p.eta * p.eta,
                 inv_dx2,     p.lambda,     p.m2,                                                   p.dx * p.dx * p.dx};
}

// Exact FP32 -> FP64 widening on the integer pipe, without a branch.  This GPU converts on its
// FP64 pipe, which the FP64 sums already keep busy: the 8 conversions per component-site of
// FP32 storage made the FP64 energy of FP32 data 1.4x slower than that of FP64 data.  Widening
// re-biases the exponent (bias 127 -> 1023) and moves the 23-bit significand to the top of the
// 52-bit one.  A subnormal (leading bit n places below the implicit one) is first shifted up by
// n and its exponent lowered by n; infinities and NaN keep the all-ones exponent, a NaN comes
// back quiet with its payload; a signed zero keeps only its sign.  The result is the one exact
// double (IEEE 754 widening), so FP64 and FP32 storage of the same values give the same sums.
__device__ __forceinline__ double widen(double v) { return v; }
__device__ __forceinline__ double widen(float v) {
    const unsigned u = __float_as_uint(v), mag = u & 0x7fffffffu;
    const int n = max(__clz(mag) - 8, 0);  // 0 for normal numbers, infinities and NaN
    const unsigned m = mag << n;
    unsigned hi = (m >> 3) + ((896u - (unsigned)n) << 20);
    hi += mag >= 0x7f800000u ? 896u << 20 : 0u;
    hi |= mag > 0x7f800000u ? 1u << 19 : 0u;
    hi = (mag ? hi : 0u) | (u & 0x80000000u);
    return __hiloint2double((int)hi, (int)(m << 29));
}

// ------------------------------------------------------------------ per-site update
// Neighbour values are passed in the fixed order -x, +x, -y, +y, -z, +z.

// Sum of the six neighbours of a site, FP64, on the integer pipes.
//
// Bound: every FP64 leapfrog and energy kernel is bound by the FP64 pipe, 2 lanes a clock per SM
// (a DADD holds it for 19 clocks a warp, a DFMA for 16), while the integer pipes, 64 + 64 lanes a
// clock, sit idle next to it and issue in its shadow (16 integer instructions beside each DFMA cost
// no time).  Five of a real site's ten FP64 instructions, and ten of a complex site's nineteen, are
// the additions of this sum, so they are done in integers instead: 256^3 complex FP64 step
// 596 -> 318 us in four-row tiles (302 in two-row ones: FP64 pipe 81 %, ALU 74 % busy), energy of
// 512^3 real FP32 storage 4.99 -> 3.79 ms.
//
// The six significands are put on one fixed-point grid, 7 bits below the last bit of the largest
// operand (unit 2^(E - 1082), E its exponent field), bits below the grid are dropped from the
// magnitudes, the 64-bit integers are added exactly, and the sum is rounded once to nearest even.
// |error| <= half an ulp of the result + 6 units, against up to half an ulp of each of five partial
// sums for additions in FP64.  The result does not depend on the operands' order and changes sign
// with them.  On Gaussian values the rms error over the largest operand is 7.0e-17, that of the addition
// tree 1.2e-16.  One class of sums is worse: where the largest operands cancel exactly, the tree keeps
// the small ones whole and this cuts them at 2^-59 of the largest (an x-pair that cancels, the others at
// 1e-6 of it: rms 1.5e-18 of the largest against 4e-20), which is below the rounding of the largest
// operands themselves.  Operands outside the grid's range (E < 64: below 2^-959; E >= 2040: huge,
// infinite or NaN) are added in FP64.
__device__ __forceinline__ unsigned long long shr_clamped(unsigned long long v, unsigned n) {
    unsigned long long r;
    asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(v), "r"(n));  // shifts of 64 and more give 0
    return r;
}

// acc (|acc| < 2^63) times 2^(x0 - 1086), rounded once to nearest even; +0 for 0.  The exponent field
// of the result, x0 - (leading zeros of |acc|), must lie in the normal range.
__device__ __forceinline__ double round_fixed(unsigned long long acc, int x0) {
    const int sign = (int)(acc >> 32) >> 31;
    const unsigned long long n0 = (acc ^ (unsigned long long)(long long)sign) - (unsigned long long)(long long)sign;
    const int lz = __clzll((long long)n0);  // 1 to 63, or 64 for 0
    const unsigned long long n = n0 << (lz - 1);  // leading bit at 62: 10 bits below the 53
    const unsigned long long r = (n + 0x1ffu + ((n >> 10) & 1u)) >> 10;
    const unsigned hi = (unsigned)(r >> 32) + ((unsigned)(x0 - 1 - lz) << 20);  // the hidden bit adds 1
    return n0 ? __hiloint2double((int)(hi | ((unsigned)sign & 0x80000000u)), (int)(unsigned)r) : 0.0;
}

// The sum in FP64.  A function of its own: inlined, its five additions were issued under a false
// predicate for every site and still held the FP64 pipe.
static __device__ __noinline__ double sum6_fp64(double a, double b, double c, double d, double e, double f) {
    return __dadd_rn(__dadd_rn(a, b), __dadd_rn(__dadd_rn(c, d), __dadd_rn(e, f)));
}

__device__ __forceinline__ double sum6(double a, double b, double c, double d, double e, double f) {
    const double v[6] = {a, b, c, d, e, f};
    unsigned mag[6];
#pragma unroll
    for (int i = 0; i < 6; ++i) mag[i] = (unsigned)__double2hiint(v[i]) & 0x7fffffffu;
    const unsigned E = __vimax3_u32(__vimax3_u32(mag[0], mag[1], mag[2]), __vimax3_u32(mag[3], mag[4], mag[5]), 0u) >> 20;
    if (E - 64u >= 2040u - 64u) {
        // six zeros, which a vacuum or a zero component has at every site, need no FP64: -0 if all are
        // (256x256x128 complex FP64 step in a vacuum of zeros 308 -> 150 us, Gaussian values 159; as a
        // function that calls sum6_fp64 this cost the multi-step kernel 2 to 6 %)
        int any = 0, all = -1;
#pragma unroll
        for (int i = 0; i < 6; ++i) {
            any |= __double2hiint(v[i]) << 1 | __double2loint(v[i]);
            all &= __double2hiint(v[i]);
        }
        return any ? sum6_fp64(a, b, c, d, e, f) : __hiloint2double(all, 0);
    }
    unsigned long long acc = 0;
#pragma unroll
    for (int i = 0; i < 6; ++i) {
        const int hi = __double2hiint(v[i]);
        const unsigned lo = (unsigned)__double2loint(v[i]);
        // 53-bit significand << 7; an exponent field of 0 is at least 64 below E and shifts out
        const unsigned mh = ((unsigned)hi & 0x000fffffu) | 0x00100000u;
        const unsigned long long m = shr_clamped((((unsigned long long)mh << 32) | lo) << 7, E - (mag[i] >> 20));
        const long long s = (long long)(hi >> 31);
        acc += (m ^ (unsigned long long)s) - (unsigned long long)s;  // +-m
    }
    return round_fixed(acc, (int)E + 4);
}

// FP64 kick (+ drift).  pi <- pi + dt F(phi);  phi_out <- phi + dt pi.
// nb: the neighbour sums (sum6) of the site's components.
template <int NC>
__device__ __forceinline__ void update_f64_nb(const double (&c)[NC], const double (&nb)[NC], double (&p)[NC],
                                              double (&out)[NC], const Coef64 &k) {
    double s2 = __dmul_rn(c[0], c[0]);
#pragma unroll
    for (int b = 1; b < NC; ++b) s2 = __fma_rn(c[b], c[b], s2);
    const double g = __fma_rn(k.dl, s2, k.b0);
#pragma unroll
    for (int a = 0; a < NC; ++a) {
        p[a] = __fma_rn(k.a, nb[a], __fma_rn(-g, c[a], p[a]));
        out[a] = __fma_rn(k.dt, p[a], c[a]);
    }
}

template <int NC>
__device__ __forceinline__ void neighbour_sums(const double (&xm)[NC], const double (&xp)[NC], const double (&ym)[NC],
                                               const double (&yp)[NC], const double (&zm)[NC], const double (&zp)[NC],
                                               double (&nb)[NC]) {
#pragma unroll
    for (int a = 0; a < NC; ++a) nb[a] = sum6(xm[a], xp[a], ym[a], yp[a], zm[a], zp[a]);
}

template <int NC>
__device__ __forceinline__ void update_f64(const double (&c)[NC], const double (&xm)[NC], const double (&xp)[NC],
                                           const double (&ym)[NC], const double (&yp)[NC], const double (&zm)[NC],
                                           const double (&zp)[NC], double (&p)[NC], double (&out)[NC],
                                           const Coef64 &k) {
    double nb[NC];
    neighbour_sums<NC>(xm, xp, ym, yp, zm, zp, nb);
    update_f64_nb<NC>(c, nb, p, out, k);
}

// FP32 force, difference form.
template <int NC>
__device__ __forceinline__ void force_f32(const float (&c)[NC], const float (&xm)[NC], const float (&xp)[NC],
                                          const float (&ym)[NC], const float (&yp)[NC], const float (&zm)[NC],
                                          const float (&zp)[NC], float (&F)[NC], const Coef32 &k) {
    float s2 = __fmul_rn(c[0], c[0]);
#pragma unroll
    for (int b = 1; b < NC; ++b) s2 = __fmaf_rn(c[b], c[b], s2);
    const float g = __fmaf_rn(k.lam, __fsub_rn(s2, k.eta2), k.m2);
#pragma unroll
    for (int a = 0; a < NC; ++a) {
        const float dx_ = __fadd_rn(__fsub_rn(xm[a], c[a]), __fsub_rn(xp[a], c[a]));
        const float dy_ = __fadd_rn(__fsub_rn(ym[a], c[a]), __fsub_rn(yp[a], c[a]));
        const float dz_ = __fadd_rn(__fsub_rn(zm[a], c[a]), __fsub_rn(zp[a], c[a]));
        const float d = __fadd_rn(__fadd_rn(dx_, dy_), dz_);
        F[a] = __fmaf_rn(d, k.inv_dx2, -__fmul_rn(g, c[a]));
    }
}

// FP32 kick + drift; KAHAN selects the compensated drift
//   y = dt pi - comp;  t = phi + y;  comp = (t - phi) - y;  phi_out = t.
template <int NC, bool KAHAN>
__device__ __forceinline__ void update_f32(const float (&c)[NC], const float (&xm)[NC], const float (&xp)[NC],
                                           const float (&ym)[NC], const float (&yp)[NC], const float (&zm)[NC],
                                           const float (&zp)[NC], float (&p)[NC], float (&cmp)[NC],
                                           float (&out)[NC], const Coef32 &k) {
    float F[NC];
    force_f32<NC>(c, xm, xp, ym, yp, zm, zp, F, k);
#pragma unroll
    for (int a = 0; a < NC; ++a) {
        p[a] = __fmaf_rn(k.dt, F[a], p[a]);
        if (KAHAN) {
            const float y = __fmaf_rn(k.dt, p[a], -cmp[a]);
            const float t = __fadd_rn(c[a], y);
            cmp[a] = __fsub_rn(__fsub_rn(t, c[a]), y);
            out[a] = t;
        } else {
            out[a] = __fmaf_rn(k.dt, p[a], c[a]);
        }
    }
}

// FP64 kick only (start of the staggered scheme): pi <- pi + dt' F(phi).
template <int NC>
__device__ __forceinline__ void kick_f64(const double (&c)[NC], const double (&xm)[NC], const double (&xp)[NC],
                                         const double (&ym)[NC], const double (&yp)[NC], const double (&zm)[NC],
                                         const double (&zp)[NC], double (&p)[NC], const Coef64 &k) {
    double out[NC];
    update_f64<NC>(c, xm, xp, ym, yp, zm, zp, p, out, k);
}

template <int NC>
__device__ __forceinline__ void kick_f32(const float (&c)[NC], const float (&xm)[NC], const float (&xp)[NC],
                                         const float (&ym)[NC], const float (&yp)[NC], const float (&zm)[NC],
                                         const float (&zp)[NC], float (&p)[NC], const Coef32 &k) {
    float F[NC];
    force_f32<NC>(c, xm, xp, ym, yp, zm, zp, F, k);
#pragma unroll
    for (int a = 0; a < NC; ++a) p[a] = __fmaf_rn(k.dt, F[a], p[a]);
}

// ------------------------------------------------------- packed FP32 pairs (f32x2)
// Two sites updated by one instruction stream with Blackwell's packed f32x2 arithmetic.
// Each lane is an IEEE round-to-nearest FP32 operation, and the sequence below is the one of
// force_f32 / update_f32 rewritten with exact sign identities of round-to-nearest
// (RN(-a*b - c) = -RN(a*b + c)), so a packed update is bitwise equal to two scalar ones.
// One caution, found by measurement: the assembler may fuse a packed multiply whose result
// feeds a packed add or subtract into a single fused multiply-add (one rounding instead of
// two) even with explicit .rn.  No product below feeds an add: c*c is formed as
// fma(c, c, zero) with a zero the compiler cannot see (RN(c*c + 0) = RN(c*c) for every c),
// and the other products feed the addend of an fma, which cannot be fused further.
typedef unsigned long long f32x2;

__device__ __forceinline__ f32x2 pk2(float lo, float hi) {
    f32x2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void up2(f32x2 v, float &lo, float &hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
    f32x2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f32x2 sub2(f32x2 a, f32x2 b) {
    f32x2 r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
    f32x2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
    f32x2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}

// Coefficients broadcast to both lanes; n* are negated copies.
struct Coef32x2 {
    f32x2 inv_dx2, nlam, eta2, nm2, dt, ndt, zero;
};

// `zero` must be a run-time 0 (the caller passes a kernel argument), never a literal.
__device__ __forceinline__ Coef32x2 make_coef32x2(const Coef32 &k, float zero) {
    return Coef32x2{pk2(k.inv_dx2, k.inv_dx2), pk2(-k.lam, -k.lam), pk2(k.eta2, k.eta2), pk2(-k.m2, -k.m2),
                    pk2(k.dt, k.dt),           pk2(-k.dt, -k.dt),   pk2(zero, zero)};
}

// update_f32 for two sites at once (lane 0 and lane 1 of every operand).
template <int NC, bool KAHAN>
__device__ __forceinline__ void update_f32x2(const f32x2 (&c)[NC], const f32x2 (&xm)[NC], const f32x2 (&xp)[NC],
                                             const f32x2 (&ym)[NC], const f32x2 (&yp)[NC], const f32x2 (&zm)[NC],
                                             const f32x2 (&zp)[NC], f32x2 (&p)[NC], f32x2 (&cmp)[NC],
                                             f32x2 (&out)[NC], const Coef32x2 &k) {
    f32x2 s2 = fma2(c[0], c[0], k.zero);
#pragma unroll
    for (int b = 1; b < NC; ++b) s2 = fma2(c[b], c[b], s2);
    const f32x2 ng = fma2(k.nlam, sub2(s2, k.eta2), k.nm2);  // -g
#pragma unroll
    for (int a = 0; a < NC; ++a) {
        const f32x2 dx_ = add2(sub2(xm[a], c[a]), sub2(xp[a], c[a]));
        const f32x2 dy_ = add2(sub2(ym[a], c[a]), sub2(yp[a], c[a]));
        const f32x2 dz_ = add2(sub2(zm[a], c[a]), sub2(zp[a], c[a]));
        const f32x2 d = add2(add2(dx_, dy_), dz_);
        const f32x2 F = fma2(d, k.inv_dx2, mul2(ng, c[a]));  // d/dx^2 - g c
        p[a] = fma2(k.dt, F, p[a]);
        if (KAHAN) {
            const f32x2 ny = fma2(k.ndt, p[a], cmp[a]);  // -(dt p - comp)
            const f32x2 t = sub2(c[a], ny);
            cmp[a] = add2(sub2(t, c[a]), ny);
            out[a] = t;
        } else {
            out[a] = fma2(k.dt, p[a], c[a]);
        }
    }
}

// update_f32 for one two-component site, its components packed as one f32x2 pair (the
// interleaved storage order): |phi|^2 and the potential coefficient are formed in scalar
// exactly as force_f32 does, everything per component runs packed.
template <bool KAHAN>
__device__ __forceinline__ void update_f32_site2(f32x2 c, f32x2 xm, f32x2 xp, f32x2 ym, f32x2 yp, f32x2 zm, f32x2 zp,
                                                 f32x2 &p, f32x2 &cmp, f32x2 &out, const Coef32x2 &k,
                                                 const Coef32 &ks) {
    float c0, c1;
    up2(c, c0, c1);
    const float s2 = __fmaf_rn(c1, c1, __fmul_rn(c0, c0));
    const float ngs = __fmaf_rn(-ks.lam, __fsub_rn(s2, ks.eta2), -ks.m2);  // -g
    const f32x2 ng = pk2(ngs, ngs);
    const f32x2 dx_ = add2(sub2(xm, c), sub2(xp, c));
    const f32x2 dy_ = add2(sub2(ym, c), sub2(yp, c));
    const f32x2 dz_ = add2(sub2(zm, c), sub2(zp, c));
    const f32x2 d = add2(add2(dx_, dy_), dz_);
    const f32x2 F = fma2(d, k.inv_dx2, mul2(ng, c));
    p = fma2(k.dt, F, p);
    if (KAHAN) {
        const f32x2 ny = fma2(k.ndt, p, cmp);
        const f32x2 t = sub2(c, ny);
        cmp = add2(sub2(t, c), ny);
        out = t;
    } else {
        out = fma2(k.dt, p, c);
    }
}

// update_f32 for one site of NC >= 3 components: |phi|^2 and the potential coefficient in
// scalar exactly as force_f32 forms them, the components in packed pairs (0,1), (2,3), ...
// with update_f32_site2's per-component sequence, and an odd last component in scalar with
// update_f32's own sequence (-g c = RN(ng * c) since ng = -g exactly).
template <int NC, bool KAHAN>
__device__ __forceinline__ void update_f32_siteN(const float (&c)[NC], const float (&xm)[NC], const float (&xp)[NC],
                                                 const float (&ym)[NC], const float (&yp)[NC], const float (&zm)[NC],
                                                 const float (&zp)[NC], float (&p)[NC], float (&cmp)[NC],
                                                 float (&out)[NC], const Coef32x2 &k, const Coef32 &ks) {
    float s2 = __fmul_rn(c[0], c[0]);
#pragma unroll
    for (int b = 1; b < NC; ++b) s2 = __fmaf_rn(c[b], c[b], s2);
    const float ngs = __fmaf_rn(-ks.lam, __fsub_rn(s2, ks.eta2), -ks.m2);  // -g
    const f32x2 ng = pk2(ngs, ngs);
#pragma unroll
    for (int q = 0; q < NC / 2; ++q) {
        const int a0 = 2 * q, a1 = 2 * q + 1;
        const f32x2 C = pk2(c[a0], c[a1]);
        const f32x2 dx_ = add2(sub2(pk2(xm[a0], xm[a1]), C), sub2(pk2(xp[a0], xp[a1]), C));
        const f32x2 dy_ = add2(sub2(pk2(ym[a0], ym[a1]), C), sub2(pk2(yp[a0], yp[a1]), C));
        const f32x2 dz_ = add2(sub2(pk2(zm[a0], zm[a1]), C), sub2(pk2(zp[a0], zp[a1]), C));
        const f32x2 d = add2(add2(dx_, dy_), dz_);
        const f32x2 F = fma2(d, k.inv_dx2, mul2(ng, C));
        f32x2 P = fma2(k.dt, F, pk2(p[a0], p[a1]));
        f32x2 O;
        if (KAHAN) {
            const f32x2 ny = fma2(k.ndt, P, pk2(cmp[a0], cmp[a1]));
            const f32x2 t = sub2(C, ny);
            up2(add2(sub2(t, C), ny), cmp[a0], cmp[a1]);
            O = t;
        } else {
            O = fma2(k.dt, P, C);
        }
        up2(P, p[a0], p[a1]);
        up2(O, out[a0], out[a1]);
    }
    if constexpr (NC % 2 == 1) {
        constexpr int a = NC - 1;
        const float dx_ = __fadd_rn(__fsub_rn(xm[a], c[a]), __fsub_rn(xp[a], c[a]));
        const float dy_ = __fadd_rn(__fsub_rn(ym[a], c[a]), __fsub_rn(yp[a], c[a]));
        const float dz_ = __fadd_rn(__fsub_rn(zm[a], c[a]), __fsub_rn(zp[a], c[a]));
        const float d = __fadd_rn(__fadd_rn(dx_, dy_), dz_);
        const float F = __fmaf_rn(d, ks.inv_dx2, __fmul_rn(ngs, c[a]));
        p[a] = __fmaf_rn(ks.dt, F, p[a]);
        if (KAHAN) {
            const float y = __fmaf_rn(ks.dt, p[a], -cmp[a]);
            const float t = __fadd_rn(c[a], y);
            cmp[a] = __fsub_rn(__fsub_rn(t, c[a]), y);
            out[a] = t;
        } else {
            out[a] = __fmaf_rn(ks.dt, p[a], c[a]);
        }
    }
}

// ----------------------------------------------------------------- geometry helpers
struct Geom {
    int nx, ny, nz;
    long long sites;
};

// The coordinates of the sites s, s + stride, s + 2 stride, ... that a thread of a grid-stride loop
// visits.  The stride is split into (x, y, z) once on the host, so a step is three additions with
// carries; two 64-bit divisions per site (about 150 instructions) took most of the issue slots of
// the per-site kernels (a step of k_site on 257 x 193 x 161 real FP32+Kahan: 53.3 -> 45.5 us; of the
// multi-step step + energy on 32^3 real FP64: 5.59 -> 5.36 us).
struct Stride3 {
    int x, y, z;
    long long sites;
};

inline Stride3 make_stride3(long long stride, const Geom &g) {
    const long long r = stride / g.nx;
    return Stride3{(int)(stride % g.nx), (int)(r % g.ny), (int)(r / g.ny), stride};
}

struct SiteWalk {
    int x, y, z;
    long long s;
    __host__ __device__ __forceinline__ SiteWalk(long long first, const Geom &g) : s(first) {
        if (first < (1LL << 31)) {
            const unsigned f = (unsigned)first, r = f / (unsigned)g.nx;
            x = (int)(f - r * (unsigned)g.nx);
            z = (int)(r / (unsigned)g.ny);
            y = (int)(r - (unsigned)z * (unsigned)g.ny);
        } else {
            const long long r = first / g.nx;
            x = (int)(first - r * g.nx);
            z = (int)(r / g.ny);
            y = (int)(r - (long long)z * g.ny);
        }
    }
    // Unsigned: a coordinate and its step are each below a side, which may be up to 2^31 - 1.
    __host__ __device__ __forceinline__ void advance(const Stride3 &d, const Geom &g) {
        s += d.sites;
        unsigned ux = (unsigned)x + (unsigned)d.x, uy = (unsigned)y + (unsigned)d.y, uz = (unsigned)z + (unsigned)d.z;
        if (ux >= (unsigned)g.nx) {
            ux -= (unsigned)g.nx;
            ++uy;
        }
        if (uy >= (unsigned)g.ny) {
            uy -= (unsigned)g.ny;
            ++uz;
        }
        x = (int)ux;
        y = (int)uy;
        z = (int)uz;  // at least nz once s is past the last site
    }
};

// The x- and y-neighbours of site i of a z-plane of fewer than 2^31 sites.
struct PlaneNbr {
    int xm, xp, ym, yp;
    __host__ __device__ __forceinline__ PlaneNbr(int i, const Geom &g) {
        const int plane = g.nx * g.ny, y = i / g.nx, x = i - y * g.nx;
        xm = x == 0 ? i - 1 + g.nx : i - 1;
        xp = x == g.nx - 1 ? i + 1 - g.nx : i + 1;
        ym = y == 0 ? i - g.nx + plane : i - g.nx;
        yp = y == g.ny - 1 ? x : i + g.nx;
    }
};

__device__ __forceinline__ int wrap_dn(int i, int n) { return i == 0 ? n - 1 : i - 1; }
__device__ __forceinline__ int wrap_up(int i, int n) { return i == n - 1 ? 0 : i + 1; }

}  // namespace lf2
