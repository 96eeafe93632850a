// lf2_energy.cu -- FP64 energy and checksum reduction (all precisions), alone or fused into a
// leapfrog step.
//
// Energy at integer step n from phi_n and pi_{n-1/2}:
//   pi_n       = pi_{n-1/2} + (dt/2) F(phi_n)          (synchronised momentum: a half kick)
//   kinetic    = sum_x 1/2 sum_a pi_{a,n}^2
//   gradient   = sum_x sum_a sum_i (phi_a(x+i) - phi_a(x))^2 / (2 dx^2)
//                (forward differences: the discrete gradient energy whose variation is the
//                 7-point Laplacian built from the Site neighbours x+i, x-i of Sec. 3.4)
//   potential  = sum_x [lambda/4 (|phi|^2 - eta^2)^2 + m2/2 |phi|^2]
// plus sum_x phi_a and sum_x phi_a^2, all times the volume element dx^3 except the sums.
//
// Each site adds raw sums (pi_n^2, squared differences, (|phi|^2 - eta^2)^2, phi_a, phi_a^2)
// to per-thread FP64 accumulators; the constant factors are applied once to the totals
// (the potential's mass term is m2/2 times the sum of the phi_a^2 totals).  A grid-stride
// pass over sites leaves one partial row per block; the last block to finish (counted with
// an atomic) sums the rows in block order and writes the record.  The grid depends only on
// the lattice and every sum has a fixed order, so the result is bitwise reproducible, and the
// fused step kernels, which visit the sites in the same order with the same per-site
// arithmetic, give bitwise the record of the stand-alone reduction.
#include <mutex>

#include "lf2_barrier.cuh"
#include "lf2_bounds.cuh"
#include "lf2_internal.cuh"

namespace lf2 {
namespace {

// Raw sums per thread for NC components: 0 kinetic, 1 gradient, 2 potential, then sum_x phi_a
// (3 + a) and sum_x phi_a^2 (3 + NC + a).  Partial rows in the scratch keep kEnergySlots
// doubles of which the first kNs<NC> are used.
template <int NC>
constexpr int kNs = 3 + 2 * NC;
// Resident blocks per SM that the kernels' registers allow: four for one component (64 registers),
// two for more (128).  The full grid is four blocks per SM, so four or two resident blocks run it in
// whole waves, where three leave the fourth block alone on its SM (256^3 real FP32 energy with 72
// registers: 470 us, with 64: 387 us).  5 and 6 components would take up to 185 registers by
// themselves, one block per SM.  At 128 FP64 spills (up to 168 bytes) and gains all the same: energy of
// 160^3, one block and two: 5 components FP64 586 and 431 us, FP32 536 and 386; 6 components 686 and 551,
// 636 and 457; FP64 step with energy 715 and 537, 849 and 671.  The multi-step launch counts on two.
template <int NC>
constexpr int kEnergyResident = NC == 1 ? 4 : 2;
constexpr int kKin = 0, kGrad = 1, kPot = 2, kSum = 3;

// L2 loads (COHERENT) where other blocks of the same launch wrote the data; the read-only
// path otherwise.  The values are the same either way.
template <bool COHERENT, typename R>
__device__ __forceinline__ R ld_field(const R *p) {
    if constexpr (COHERENT)
        return __ldcg(p);
    else
        return __ldg(p);
}

template <typename R, int NC, bool COHERENT = false>
__device__ __forceinline__ void load_site(const R *__restrict__ f, long long s, long long sites, R (&v)[NC]) {
    const long long i = checked(s * NC, NC, sites * NC);
#pragma unroll
    for (int a = 0; a < NC; ++a) v[a] = ld_field<COHERENT>(f + i + a);
}

// --------------------------------------- sums and differences of the energy, in integers
// The FP64 pipe bounds the energy kernels while the integer pipes have time left (see sum6), so the
// forward differences are subtracted as integers too: both significands on one grid, an exact
// difference, rounded once.  FP32 values are widened for the FP64 energy, and their neighbour sums
// and differences are taken directly from the FP32 words: each operand is its signed 24-bit
// significand times a power of two, one wide multiply-add.  All bit for bit the FP64 operations on
// the (widened) values; operands outside a fast range (orders of magnitude apart, tiny, huge,
// infinite, NaN) take those, in functions of their own so that their instructions are not issued
// under a false predicate.  FP32 zeros, exact too, come to those functions but need no FP64 operation
// (256x256x128 complex FP32 energy: a zero component 456 -> 332 us, a lump in a vacuum of zeros 582 ->
// 329); FP64 zeros need none in the sums (sum6), but in the differences, where the test for them made
// the energy of 5 and 6 components 3 % slower.
// 256^3, one energy: 1 component FP64 476 -> 390 us, 2 components 811 -> 718 (differences);
// FP32 storage 485 -> 387 and 854 -> 657 us (sums and differences).
__device__ __noinline__ double sum6_widened(float a, float b, float c, float d, float e, float f) {
    const float v[6] = {a, b, c, d, e, f};
    int any = 0, all = -1;
#pragma unroll
    for (int i = 0; i < 6; ++i) {
        any |= __float_as_int(v[i]) << 1;
        all &= __float_as_int(v[i]);
    }
    if (!any) return __hiloint2double(all, 0);  // -0 if all are, else +0
    return sum6(widen(a), widen(b), widen(c), widen(d), widen(e), widen(f));
}
__device__ __noinline__ double sub_fp64(double a, double b) { return __dsub_rn(a, b); }
__device__ __noinline__ double sub_widened(float a, float b) {
    const int ua = __float_as_int(a), ub = __float_as_int(b);
    if (!(ub << 1)) return ua << 1 ? widen(a) : __hiloint2double(ua & ~ub & (int)0x80000000, 0);
    if (!(ua << 1)) return widen(-b);
    return sub_fp64(widen(a), widen(b));
}

// The signed 24-bit significand of a normal number.
__device__ __forceinline__ int significand(float v) {
    const int u = __float_as_int(v), s = u >> 31;
    return (((u & 0x007fffff) | 0x00800000) ^ s) - s;
}
__device__ __forceinline__ unsigned magnitude(float v) { return __float_as_uint(v) & 0x7fffffffu; }
// 2^n for n in 0..31, 0 for any other n (as unsigned)
__device__ __forceinline__ int pow2_clamped(unsigned n) {
    int r;
    asm("shl.b32 %0, 1, %1;" : "=r"(r) : "r"(n));
    return r;
}

__device__ __forceinline__ double neighbour_sum(double a, double b, double c, double d, double e, double f) {
    return sum6(a, b, c, d, e, f);
}
__device__ __forceinline__ double neighbour_sum(float a, float b, float c, float d, float e, float f) {
    const float v[6] = {a, b, c, d, e, f};
    unsigned m[6];
#pragma unroll
    for (int i = 0; i < 6; ++i) m[i] = magnitude(v[i]);
    const unsigned hi = __vimax3_u32(__vimax3_u32(m[0], m[1], m[2]), __vimax3_u32(m[3], m[4], m[5]), 0u);
    // the smallest but for zeros, which wrap to the largest and contribute nothing below
    const unsigned lo = __vimin3_u32(__vimin3_u32(m[0] - 1u, m[1] - 1u, m[2] - 1u),
                                     __vimin3_u32(m[3] - 1u, m[4] - 1u, m[5] - 1u), 0xffffffffu);
    const unsigned E = hi >> 23;
    // m - 1 may have an exponent one lower: 29 binary orders keep every operand within 30
    if (E - 32u >= 255u - 32u || (lo >> 23) + 29u < E) return sum6_widened(a, b, c, d, e, f);
    long long acc = 0;
#pragma unroll
    for (int i = 0; i < 6; ++i) acc += (long long)significand(v[i]) * pow2_clamped(30u - E + (m[i] >> 23));
    return round_fixed((unsigned long long)acc, (int)E + 906);
}

// a - b, exact in FP64 when the exponents are at most 28 apart.
__device__ __forceinline__ double sub_exact(float a, float b) {
    const unsigned ma = magnitude(a), mb = magnitude(b);
    const unsigned E = max(ma, mb) >> 23, F = min(ma, mb) >> 23;
    if (F - 1u >= 254u || E == 255u || F + 28u < E) return sub_widened(a, b);  // F = 0: zero or subnormal
    const unsigned long long d = (unsigned long long)((long long)significand(a) * pow2_clamped(28u - E + (ma >> 23)) -
                                                      (long long)significand(b) * pow2_clamped(28u - E + (mb >> 23)));
    const int sign = (int)(d >> 32) >> 31;
    const unsigned long long n0 = (d ^ (unsigned long long)(long long)sign) - (unsigned long long)(long long)sign;
    const int lz = __clzll((long long)n0);        // 11 to 63, or 64 for 0
    const unsigned long long n = n0 << (lz - 11);  // leading bit at 52, nothing to round
    const unsigned hi = (unsigned)(n >> 32) + ((E + 907u - (unsigned)lz) << 20);
    return n0 ? __hiloint2double((int)(hi | ((unsigned)sign & 0x80000000u)), (int)(unsigned)n) : 0.0;
}
// FP64: with exponents at most 9 apart no bit is lost and the difference stays below 2^63.
__device__ __forceinline__ double sub_exact(double a, double b) {
    const int ha = __double2hiint(a), hb = __double2hiint(b);
    const unsigned ma = (unsigned)ha & 0x7fffffffu, mb = (unsigned)hb & 0x7fffffffu;
    const unsigned E = max(ma, mb) >> 20, F = min(ma, mb) >> 20;
    if (E - 64u >= 2040u - 64u || F + 9u < E) return sub_fp64(a, b);
    const unsigned long long A = (((unsigned long long)((ma & 0x000fffffu) | 0x00100000u) << 32) |
                                  (unsigned)__double2loint(a)) << (9u - E + (ma >> 20));
    const unsigned long long B = (((unsigned long long)((mb & 0x000fffffu) | 0x00100000u) << 32) |
                                  (unsigned)__double2loint(b)) << (9u - E + (mb >> 20));
    const unsigned long long sa = (unsigned long long)(long long)(ha >> 31), sb = (unsigned long long)(long long)(~hb >> 31);
    return round_fixed((A ^ sa) + (B ^ sb) - sa - sb, (int)E + 2);
}

// Adds one site's raw sums to acc.  c: phi_n at the site, xm..zp: its neighbours in the order
// -x, +x, -y, +y, -z, +z; p: pi_{n-1/2}, in the storage type.  Explicit round-to-nearest
// operations keep the stand-alone and fused kernels bitwise equal; the half kick is the FP64 kick's
// arithmetic.  Component by component, so that few widened values are live at once.  nb: the
// neighbour sums, which the FP64 update uses too; computed here unless HAVE_NB.  INTSUB: the
// differences in integers (the multi-step kernel's FP64 instance, bound by latency, is 3 % faster
// with FP64 subtractions).
template <typename R, int NC, bool INTSUB, bool HAVE_NB = false>
__device__ __forceinline__ void energy_site(const R (&c)[NC], const R (&xm)[NC], const R (&xp)[NC], const R (&ym)[NC],
                                            const R (&yp)[NC], const R (&zm)[NC], const R (&zp)[NC], const R (&p)[NC],
                                            double (&nb)[NC], double (&acc)[kNs<NC>], const CoefE &k) {
    double s2;
    {
        const double d = widen(c[0]);
        s2 = __dmul_rn(d, d);
    }
#pragma unroll
    for (int b = 1; b < NC; ++b) {
        const double d = widen(c[b]);
        s2 = __fma_rn(d, d, s2);
    }
    const double gh = __fma_rn(k.hl, s2, k.hb0);
    const double w = __dsub_rn(s2, k.eta2);
    acc[kPot] = __fma_rn(w, w, acc[kPot]);
#pragma unroll
    for (int a = 0; a < NC; ++a) {
        if (!HAVE_NB) nb[a] = neighbour_sum(xm[a], xp[a], ym[a], yp[a], zm[a], zp[a]);
        const double d = widen(c[a]);
        const double pin = __fma_rn(k.ah, nb[a], __fma_rn(-gh, d, widen(p[a])));
        acc[kKin] = __fma_rn(pin, pin, acc[kKin]);
        const double ex = INTSUB ? sub_exact(xp[a], c[a]) : __dsub_rn(widen(xp[a]), d);
        const double ey = INTSUB ? sub_exact(yp[a], c[a]) : __dsub_rn(widen(yp[a]), d);
        const double ez = INTSUB ? sub_exact(zp[a], c[a]) : __dsub_rn(widen(zp[a]), d);
        acc[kGrad] = __fma_rn(ez, ez, __fma_rn(ey, ey, __fma_rn(ex, ex, acc[kGrad])));
        acc[kSum + a] = __dadd_rn(acc[kSum + a], d);
        acc[kSum + NC + a] = __fma_rn(d, d, acc[kSum + NC + a]);
    }
}

// Block sum of acc, left in sh[j][0].  A pairwise tree whose additions at each level are packed
// onto consecutive threads: an FP64 warp instruction costs the same however few of its lanes
// are active, so the levels with fewer than 32 pairs per sum still fill whole warps.
template <int NS>
__device__ __forceinline__ void block_sum(const double (&acc)[NS], double (&sh)[NS][kEnergyThreads]) {
#pragma unroll
    for (int j = 0; j < NS; ++j) sh[j][threadIdx.x] = acc[j];
    __syncthreads();
#pragma unroll
    for (int w = kEnergyThreads / 2; w > 0; w >>= 1) {
        for (int t = threadIdx.x; t < NS * w; t += kEnergyThreads) {
            const int j = t / w, i = t % w;
            sh[j][i] = __dadd_rn(sh[j][i], sh[j][i + w]);
        }
        __syncthreads();
    }
}

// Sums `nrows` partial rows (L2 reads, in row order) with the block and writes the record
// (thread 0) to `record` and, when not NULL, to `own`.  All threads of the block take part.
template <int NC>
__device__ __forceinline__ void reduce_rows(const double *rows, int nrows, double (&sh)[kNs<NC>][kEnergyThreads],
                                            const CoefE &k, double *__restrict__ record, double *__restrict__ own) {
    constexpr int NS = kNs<NC>;
    double tot[NS];
#pragma unroll
    for (int j = 0; j < NS; ++j) tot[j] = 0.0;
    for (int b = threadIdx.x; b < nrows; b += blockDim.x) {
#pragma unroll
        for (int j = 0; j < NS; ++j) tot[j] = __dadd_rn(tot[j], __ldcg(rows + (size_t)b * kEnergySlots + j));
    }
    block_sum<NS>(tot, sh);
    if (threadIdx.x == 0) {
        double r[kEnergySlots];
        double ssq = 0.0;
        for (int a = 0; a < NC; ++a) ssq += sh[kSum + NC + a][0];
        r[0] = k.vol * (0.5 * sh[kKin][0]);
        r[1] = k.vol * (0.5 * k.inv_dx2 * sh[kGrad][0]);
        r[2] = k.vol * (0.25 * k.lam * sh[kPot][0] + 0.5 * k.m2 * ssq);
        r[3] = r[0] + r[1] + r[2];
        for (int a = 0; a < kMaxComp; ++a) {
            r[4 + a] = a < NC ? sh[kSum + a][0] : 0.0;
            r[4 + kMaxComp + a] = a < NC ? sh[kSum + NC + a][0] : 0.0;
        }
        for (int j = 0; j < kEnergySlots; ++j) {
            if (own) own[j] = r[j];
            if (record) record[j] = r[j];
        }
    }
}

// End of every energy kernel: stores this block's partial row, and the last block to get here
// sums all rows (in block order) and writes the record.  No block waits for another.
template <int NC>
__device__ __forceinline__ void finish_energy(const double (&acc)[kNs<NC>], double (&sh)[kNs<NC>][kEnergyThreads],
                                              double *__restrict__ scratch, const CoefE &k,
                                              double *__restrict__ record) {
    constexpr int NS = kNs<NC>;
    __shared__ bool s_last;
    block_sum<NS>(acc, sh);
    if (threadIdx.x < NS) scratch[(size_t)blockIdx.x * kEnergySlots + threadIdx.x] = sh[threadIdx.x][0];
    __threadfence();  // this block's row is visible device-wide before the block is counted
    __syncthreads();
    unsigned int *counter = reinterpret_cast<unsigned int *>(scratch + kEnergyCounterOffset);
    if (threadIdx.x == 0) s_last = atomicAdd(counter, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!s_last) return;
    __threadfence();  // every other block's row is visible to this one
    reduce_rows<NC>(scratch, (int)gridDim.x, sh, k, record, scratch + kEnergyRecordOffset);
    if (threadIdx.x == 0) *counter = 0u;  // ready for the next launch on this scratch
}

// Linear indices of the six periodic neighbours of site s.
struct Nbr {
    long long xm, xp, ym, yp, zm, zp;
};

__device__ __forceinline__ Nbr neighbours(const SiteWalk &w, const Geom &g) {
    const long long row = g.nx, plane = (long long)g.nx * g.ny;
    return Nbr{w.s + (w.x == 0 ? g.nx - 1 : -1),          w.s + (w.x == g.nx - 1 ? 1 - g.nx : 1),
               w.s + (wrap_dn(w.y, g.ny) - w.y) * row,    w.s + (wrap_up(w.y, g.ny) - w.y) * row,
               w.s + (wrap_dn(w.z, g.nz) - w.z) * plane,  w.s + (wrap_up(w.z, g.nz) - w.z) * plane};
}

template <typename R, int NC>
__global__ void __launch_bounds__(kEnergyThreads, kEnergyResident<NC>) k_energy(const R *__restrict__ phi, const R *__restrict__ pi, Geom g,
                                                           Stride3 d, CoefE k, double *__restrict__ scratch,
                                                           double *__restrict__ record) {
    __shared__ double sh[kNs<NC>][kEnergyThreads];
    double acc[kNs<NC>];
#pragma unroll
    for (int j = 0; j < kNs<NC>; ++j) acc[j] = 0.0;
    for (SiteWalk w((long long)blockIdx.x * blockDim.x + threadIdx.x, g); w.s < g.sites; w.advance(d, g)) {
        const Nbr n = neighbours(w, g);
        const long long s = w.s;
        R c[NC], xm[NC], xp[NC], ym[NC], yp[NC], zm[NC], zp[NC], p[NC];
        load_site<R, NC>(phi, s, g.sites, c);
        load_site<R, NC>(phi, n.xm, g.sites, xm);
        load_site<R, NC>(phi, n.xp, g.sites, xp);
        load_site<R, NC>(phi, n.ym, g.sites, ym);
        load_site<R, NC>(phi, n.yp, g.sites, yp);
        load_site<R, NC>(phi, n.zm, g.sites, zm);
        load_site<R, NC>(phi, n.zp, g.sites, zp);
        load_site<R, NC>(pi, s, g.sites, p);
        double nb[NC];
        energy_site<R, NC, true>(c, xm, xp, ym, yp, zm, zp, p, nb, acc, k);
    }
    finish_energy<NC>(acc, sh, scratch, k, record);
}

// One site of a fused step + energy, FP64: adds the energy of (phi_n, pi_{n-1/2}) at site s
// to acc and writes the step to (phi_{n+1}, pi_{n+1/2}), from one read of the site's stencil.
template <int NC>
__device__ __forceinline__ void site_step_energy_f64(const double *__restrict__ phi, double *__restrict__ phi_out,
                                                     double *__restrict__ pi, const SiteWalk &w, const Geom &g,
                                                     const Coef64 &k, const CoefE &ke, double (&acc)[kNs<NC>]) {
    const Nbr n = neighbours(w, g);
    const long long s = w.s;
    double c[NC], xm[NC], xp[NC], ym[NC], yp[NC], zm[NC], zp[NC], p[NC], out[NC];
    load_site<double, NC>(phi, s, g.sites, c);
    load_site<double, NC>(phi, n.xm, g.sites, xm);
    load_site<double, NC>(phi, n.xp, g.sites, xp);
    load_site<double, NC>(phi, n.ym, g.sites, ym);
    load_site<double, NC>(phi, n.yp, g.sites, yp);
    load_site<double, NC>(phi, n.zm, g.sites, zm);
    load_site<double, NC>(phi, n.zp, g.sites, zp);
    const long long o = checked(s * NC, NC, g.sites * NC);
#pragma unroll
    for (int a = 0; a < NC; ++a) p[a] = pi[o + a];
    double nb[NC];
    energy_site<double, NC, true>(c, xm, xp, ym, yp, zm, zp, p, nb, acc, ke);
    update_f64_nb<NC>(c, nb, p, out, k);
#pragma unroll
    for (int a = 0; a < NC; ++a) {
        pi[o + a] = p[a];
        phi_out[o + a] = out[a];
    }
}

// The same for FP32 storage (KAHAN: compensated drift); the energy is computed in FP64 from
// the exact conversions of the stored values.
template <int NC, bool KAHAN>
__device__ __forceinline__ void site_step_energy_f32(const float *__restrict__ phi, float *__restrict__ phi_out,
                                                     float *__restrict__ pi, float *__restrict__ comp, const SiteWalk &w,
                                                     const Geom &g, const Coef32 &k, const CoefE &ke,
                                                     double (&acc)[kNs<NC>]) {
    const Nbr n = neighbours(w, g);
    const long long s = w.s;
    const long long cnt = g.sites * NC;
    const long long o = checked(s * NC, NC, cnt), ixm = checked(n.xm * NC, NC, cnt), ixp = checked(n.xp * NC, NC, cnt),
                    iym = checked(n.ym * NC, NC, cnt), iyp = checked(n.yp * NC, NC, cnt),
                    izm = checked(n.zm * NC, NC, cnt), izp = checked(n.zp * NC, NC, cnt);
    float c[NC], xm[NC], xp[NC], ym[NC], yp[NC], zm[NC], zp[NC], p[NC], cm[NC], out[NC];
#pragma unroll
    for (int a = 0; a < NC; ++a) {
        c[a] = __ldg(phi + o + a);
        xm[a] = __ldg(phi + ixm + a);
        xp[a] = __ldg(phi + ixp + a);
        ym[a] = __ldg(phi + iym + a);
        yp[a] = __ldg(phi + iyp + a);
        zm[a] = __ldg(phi + izm + a);
        zp[a] = __ldg(phi + izp + a);
        p[a] = pi[o + a];
        cm[a] = KAHAN ? comp[o + a] : 0.0f;
    }
    double nb[NC];
    energy_site<float, NC, true>(c, xm, xp, ym, yp, zm, zp, p, nb, acc, ke);
    update_f32<NC, KAHAN>(c, xm, xp, ym, yp, zm, zp, p, cm, out, k);
#pragma unroll
    for (int a = 0; a < NC; ++a) {
        pi[o + a] = p[a];
        phi_out[o + a] = out[a];
        if (KAHAN) comp[o + a] = cm[a];
    }
}

// Fused step + energy, one step per launch.
template <int NC>
__global__ void __launch_bounds__(kEnergyThreads, kEnergyResident<NC>)
    k_step_energy_f64(const double *__restrict__ phi, double *__restrict__ phi_out, double *__restrict__ pi, Geom g,
                      Stride3 d, Coef64 k, CoefE ke, double *__restrict__ scratch, double *__restrict__ record) {
    __shared__ double sh[kNs<NC>][kEnergyThreads];
    double acc[kNs<NC>];
#pragma unroll
    for (int j = 0; j < kNs<NC>; ++j) acc[j] = 0.0;
    for (SiteWalk w((long long)blockIdx.x * blockDim.x + threadIdx.x, g); w.s < g.sites; w.advance(d, g))
        site_step_energy_f64<NC>(phi, phi_out, pi, w, g, k, ke, acc);
    finish_energy<NC>(acc, sh, scratch, ke, record);
}

// Four blocks for two components too, in spite of 84 bytes of spills and more: 160^3 FP32+Kahan 178.4 us with
// two, 176.9 with four; 96x80x112 51.1 and 50.1.  (In FP64 four are 5 % slower.)  5 and 6 components with one
// block: 574 and 702 us, with two 408 and 495.
template <int NC, bool KAHAN>
__global__ void __launch_bounds__(kEnergyThreads, NC <= 2 ? 4 : 2)
    k_step_energy_f32(const float *__restrict__ phi, float *__restrict__ phi_out, float *__restrict__ pi,
                      float *__restrict__ comp, Geom g, Stride3 d, Coef32 k, CoefE ke,
                      double *__restrict__ scratch, double *__restrict__ record) {
    __shared__ double sh[kNs<NC>][kEnergyThreads];
    double acc[kNs<NC>];
#pragma unroll
    for (int j = 0; j < kNs<NC>; ++j) acc[j] = 0.0;
    for (SiteWalk w((long long)blockIdx.x * blockDim.x + threadIdx.x, g); w.s < g.sites; w.advance(d, g))
        site_step_energy_f32<NC, KAHAN>(phi, phi_out, pi, comp, w, g, k, ke, acc);
    finish_energy<NC>(acc, sh, scratch, ke, record);
}

// ------------------------------------------- many steps in one launch (small lattices)
// On a small lattice a step is a few microseconds of launch gaps and latency around very little
// arithmetic.  One cooperative launch runs all steps, with a grid barrier (lf2_barrier.cuh) between
// them, for lattices that give every resident thread at most one site: a thread keeps its site's
// field value, momentum and compensation in registers from step to step, loads six neighbours,
// stores one field value and arrives at the barrier.  The arithmetic is the one-step kernels', so
// fields and records are bitwise those of one launch per step.
//
// ENERGY: the records of k_step_energy too, with its partial sums and their order.  The energy of a
// step comes after the arrival, while the other blocks arrive: the site blocks add it up and write
// the partial row of step k before they arrive at barrier k+1, and one extra block, which owns no
// sites, reduces the rows of step k once barrier k+1 has completed, while the site blocks run step
// k+2; one more barrier after the last step completes its rows.  The rows rotate over three sets: a
// site block writes the set of step k+3 only after barrier k+2, which the reducing block joins only
// after it has read the rows of step k.
//
// 32^3 real FP64, a step: 3.8 us with its energy (4.1 with the energy before the arrival and pi in
// memory, 5.3 with a two-atomic barrier too), 2.2 without (4.3 at best as launches of the streaming
// kernel); 48x40x36 real FP32+Kahan without energy 6.1 -> 1.8 us.  More components, without energy, as
// four-row streaming or site launches and here: 32^3 FP64, 2 components 8.3 and 3.0 us, 4: 10.4 and 4.6,
// 6: 14.5 and 6.4; 48^3 10.4 and 5.1, 16.6 and 10.4, 24.7 and 14.5; FP32+Kahan 48^3 6.3 and 2.6, 8.3 and
// 4.3, 12.4 and 6.3.  What is left is the barrier's trips through L2 and the loads that follow it.

// The row sets (at most kStepsMaxBlocks rows each) start at kStepsRowsOffset of a field's
// scratch; the barrier and status words (lf2_barrier.cuh) are in the counter's row before them.
constexpr int kRowSets = kEnergyStepsRowSets;
constexpr int kStepsMaxBlocks = kEnergyStepsBlocks;

// A run cut short by a barrier that did not complete leaves NaN records from `from` on (the
// record of a step is finished during the next step, so `from` is the step before that barrier).
__device__ __forceinline__ void poison_records(double *records, int from, int nsteps) {
    if (blockIdx.x != gridDim.x - 1 || threadIdx.x != 0) return;
    for (int j = from; j < nsteps; ++j)
        for (int i = 0; i < kEnergySlots; ++i) records[(size_t)j * kEnergySlots + i] = __longlong_as_double(0x7ff8000000000000LL);
}

// MODE: 0 = FP32 plain drift, 1 = FP32 Kahan drift, 3 = FP64.  Launched with a site block for every 256
// sites, and with ENERGY, where they are energy_grid(sites) blocks, one more.
template <typename R, int NC, int MODE, bool ENERGY, typename CoefT>
__global__ void __launch_bounds__(kEnergyThreads, 2)
    k_steps(R *phi_a, R *phi_b, R *__restrict__ pi, float *__restrict__ comp, Geom g, CoefT k, CoefE ke, int nsteps,
            double *__restrict__ scratch, double *__restrict__ records, unsigned polls) {
    constexpr int NS = kNs<NC>;
    __shared__ double sh[ENERGY ? NS : 1][ENERGY ? kEnergyThreads : 1];
    unsigned long long *bar = reinterpret_cast<unsigned long long *>(scratch + kStepsBarrierWord);
    unsigned long long *status = reinterpret_cast<unsigned long long *>(scratch + kStepsStatusWord);
    const int nsb = ENERGY ? (int)gridDim.x - 1 : (int)gridDim.x;
    const bool reducer = ENERGY && (int)blockIdx.x == nsb;
    // rows [first, first + count) of the set of `step`, inside the row-set region (checked in
    // the debug build against that region, so that nothing before or after it can be hit)
    auto rows_of = [&](int step, long long first, long long count) {
        const long long rel = checked((long long)(step % kRowSets) * nsb * kEnergySlots + first * kEnergySlots,
                                      count * kEnergySlots, (long long)kRowSets * kStepsMaxBlocks * kEnergySlots);
        return scratch + kStepsRowsOffset + rel;
    };
    const SiteWalk w((long long)blockIdx.x * kEnergyThreads + threadIdx.x, g);
    const bool active = !reducer && w.s < g.sites;
    const Nbr n = active ? neighbours(w, g) : Nbr{0, 0, 0, 0, 0, 0};
    const long long o = active ? checked(w.s * NC, NC, g.sites * NC) : 0;
    R c[NC], p[NC];
    float cm[NC];
#pragma unroll
    for (int a = 0; a < NC; ++a) {
        c[a] = active ? __ldcg(phi_a + o + a) : R(0);
        p[a] = active ? pi[o + a] : R(0);
        cm[a] = active && MODE == 1 ? comp[o + a] : 0.0f;
    }
    for (int step = 0; step < nsteps + (ENERGY ? 1 : 0); ++step) {
        const bool stepping = active && step < nsteps;
        R xm[NC], xp[NC], ym[NC], yp[NC], zm[NC], zp[NC], pn[NC], out[NC];
        double nb[NC];
        if (stepping) {
            const R *src = (step & 1) ? phi_b : phi_a;
            R *dst = (step & 1) ? phi_a : phi_b;
            load_site<R, NC, true>(src, n.xm, g.sites, xm);
            load_site<R, NC, true>(src, n.xp, g.sites, xp);
            load_site<R, NC, true>(src, n.ym, g.sites, ym);
            load_site<R, NC, true>(src, n.yp, g.sites, yp);
            load_site<R, NC, true>(src, n.zm, g.sites, zm);
            load_site<R, NC, true>(src, n.zp, g.sites, zp);
#pragma unroll
            for (int a = 0; a < NC; ++a) pn[a] = p[a];
            if constexpr (MODE == 3) {
                neighbour_sums<NC>(xm, xp, ym, yp, zm, zp, nb);
                update_f64_nb<NC>(c, nb, pn, out, k);
            } else {
                update_f32<NC, MODE == 1>(c, xm, xp, ym, yp, zm, zp, pn, cm, out, k);
            }
#pragma unroll
            for (int a = 0; a < NC; ++a) dst[o + a] = out[a];
        }
        if (!ENERGY && step == nsteps - 1) {
            if (stepping) {
#pragma unroll
                for (int a = 0; a < NC; ++a) p[a] = pn[a];
            }
            break;
        }
        grid_arrive(bar);  // step's fields published (the final pass: rows only)
        if constexpr (ENERGY) {
            if (!reducer && step < nsteps) {
                double acc[NS];
#pragma unroll
                for (int j = 0; j < NS; ++j) acc[j] = 0.0;
                if (stepping) energy_site<R, NC, MODE != 3, MODE == 3>(c, xm, xp, ym, yp, zm, zp, p, nb, acc, ke);
                block_sum<NS>(acc, sh);
                if (threadIdx.x < NS) rows_of(step, blockIdx.x, 1)[threadIdx.x] = sh[threadIdx.x][0];
            }
        }
        if (stepping) {
#pragma unroll
            for (int a = 0; a < NC; ++a) {
                c[a] = out[a];
                p[a] = pn[a];
            }
        }
        if (!grid_wait(bar, status, (step + 1ull) * gridDim.x, polls)) {
            if constexpr (ENERGY) poison_records(records, step > 0 ? step - 1 : 0, nsteps);
            return;
        }
        if constexpr (ENERGY) {
            if (reducer && step > 0)
                reduce_rows<NC>(rows_of(step - 1, 0, nsb), nsb, sh, ke, records + (size_t)(step - 1) * kEnergySlots, nullptr);
        }
    }
    if (active) {
#pragma unroll
        for (int a = 0; a < NC; ++a) {
            pi[o + a] = p[a];
            if (MODE == 1) comp[o + a] = cm[a];
        }
    }
}

// One block per 256 sites up to kEnergyBlocks: small lattices (a 32^3 run with an energy every
// step) spread over many SMs, large ones keep at most kEnergyBlocks partial rows.
int energy_grid(long long sites) {
    const long long want = (sites + kEnergyThreads - 1) / kEnergyThreads;
    return (int)(want < 1 ? 1 : (want > kEnergyBlocks ? kEnergyBlocks : want));
}

template <typename R>
cudaError_t launch_typed(const void *phi, const void *pi, const Geom &g, int ncomp, const CoefE &k, double *scratch,
                         double *record, cudaStream_t s) {
    const int nb = energy_grid(g.sites);
    const Stride3 d = make_stride3((long long)nb * kEnergyThreads, g);
    switch (ncomp) {
#define LF2_E(NC)                                                                                               \
    case NC:                                                                                                    \
        k_energy<R, NC><<<nb, kEnergyThreads, 0, s>>>((const R *)phi, (const R *)pi, g, d, k, scratch, record); \
        break;
        LF2_E(1) LF2_E(2) LF2_E(3) LF2_E(4) LF2_E(5) LF2_E(6)
#undef LF2_E
        default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

template <int NC>
void step_energy_nc(const StepArgs &a, const CoefE &ke, int nb, double *scratch, double *record, cudaStream_t s) {
    const Stride3 d = make_stride3((long long)nb * kEnergyThreads, a.g);
    if (a.prec == LF2_F64) {
        k_step_energy_f64<NC><<<nb, kEnergyThreads, 0, s>>>((const double *)a.phi, (double *)a.phi_out, (double *)a.pi,
                                                            a.g, d, make_coef64(a.p, a.dt), ke, scratch, record);
        return;
    }
    const Coef32 k = make_coef32(a.p, a.dt);
    if (a.prec == LF2_F32_KAHAN)
        k_step_energy_f32<NC, true><<<nb, kEnergyThreads, 0, s>>>((const float *)a.phi, (float *)a.phi_out,
                                                                  (float *)a.pi, a.comp, a.g, d, k, ke, scratch, record);
    else
        k_step_energy_f32<NC, false><<<nb, kEnergyThreads, 0, s>>>((const float *)a.phi, (float *)a.phi_out,
                                                                   (float *)a.pi, a.comp, a.g, d, k, ke, scratch, record);
}

// ------------------------------------------------------------ error norms (a12)
// max |a - ref|, max |ref|, sum (a - ref)^2, sum ref^2 over n elements, FP64.  The maxima
// propagate NaN (a NaN difference must not vanish from an error report).  Per element they are
// taken on the integer pipe: with the sign bit cleared, the bit patterns of doubles order as
// unsigned integers exactly as their values do, and every NaN orders above +inf, so the
// largest pattern is the largest magnitude, or a NaN if one occurred.  Only the subtraction
// and the two squares use the FP64 pipe, which bounds this kernel.
__device__ __forceinline__ double nanmax(double m, double x) { return (x > m || x != x) ? x : m; }

constexpr int kCmp = 4;

// Running maximum of |x| as its bit pattern (sign cleared), compared as the pair (high word,
// low word) in 32-bit integer operations.  (A 64-bit unsigned max here kept the FP64 pipe as
// busy as the two FP64 comparisons it replaced: 0.36 ms against 0.20 ms for this kernel on a
// 256^3 complex field.)
struct MagMax {
    unsigned hi = 0u, lo = 0u;
    __device__ __forceinline__ void add(double x) {
        const unsigned h = (unsigned)__double2hiint(x) & 0x7fffffffu, l = (unsigned)__double2loint(x);
        const bool gt = h > hi || (h == hi && l > lo);
        hi = gt ? h : hi;
        lo = gt ? l : lo;
    }
    __device__ __forceinline__ double value() const { return __hiloint2double((int)hi, (int)lo); }
};

__device__ __forceinline__ void block_cmp(const double (&acc)[kCmp], double (&sh)[kCmp][kEnergyThreads]) {
#pragma unroll
    for (int j = 0; j < kCmp; ++j) sh[j][threadIdx.x] = acc[j];
    __syncthreads();
#pragma unroll
    for (int w = kEnergyThreads / 2; w > 0; w >>= 1) {
        for (int t = threadIdx.x; t < kCmp * w; t += kEnergyThreads) {
            const int j = t / w, i = t % w;
            sh[j][i] = j < 2 ? nanmax(sh[j][i], sh[j][i + w]) : __dadd_rn(sh[j][i], sh[j][i + w]);
        }
        __syncthreads();
    }
}

template <typename RA, typename RB>
__global__ void __launch_bounds__(kEnergyThreads) k_compare(const RA *__restrict__ a, const RB *__restrict__ ref,
                                                            long long n, double *__restrict__ scratch) {
    __shared__ double sh[kCmp][kEnergyThreads];
    __shared__ bool s_last;
    double acc[kCmp] = {0.0, 0.0, 0.0, 0.0};
    MagMax max_d, max_r;
    // The thread's elements i, i + stride, i + 2 stride, ... are taken kBatch at a time: all their
    // loads are issued before the first is used (the bound checks come first, so no load is
    // speculative), and the sums still run in element order.
    constexpr int kBatch = 4;
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long i0 = (long long)blockIdx.x * blockDim.x + threadIdx.x; i0 < n; i0 += kBatch * stride) {
        RA av[kBatch];
        RB rv[kBatch];
#pragma unroll
        for (int u = 0; u < kBatch; ++u) {
            const long long i = i0 + u * stride;
            av[u] = i < n ? __ldg(a + i) : RA(0);
            rv[u] = i < n ? __ldg(ref + i) : RB(0);
        }
#pragma unroll
        for (int u = 0; u < kBatch; ++u) {
            if (i0 + u * stride >= n) break;
            const double r = widen(rv[u]);
            const double d = __dsub_rn(widen(av[u]), r);
            max_d.add(d);
            max_r.add(r);
            acc[2] = __fma_rn(d, d, acc[2]);
            acc[3] = __fma_rn(r, r, acc[3]);
        }
    }
    acc[0] = max_d.value();
    acc[1] = max_r.value();
    block_cmp(acc, sh);
    if (threadIdx.x < kCmp) scratch[(size_t)blockIdx.x * kEnergySlots + threadIdx.x] = sh[threadIdx.x][0];
    __threadfence();
    __syncthreads();
    unsigned int *counter = reinterpret_cast<unsigned int *>(scratch + kEnergyCounterOffset);
    if (threadIdx.x == 0) s_last = atomicAdd(counter, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    double tot[kCmp] = {0.0, 0.0, 0.0, 0.0};
    for (int b = threadIdx.x; b < (int)gridDim.x; b += blockDim.x) {
#pragma unroll
        for (int j = 0; j < kCmp; ++j) {
            const double v = __ldcg(scratch + (size_t)b * kEnergySlots + j);
            tot[j] = j < 2 ? nanmax(tot[j], v) : __dadd_rn(tot[j], v);
        }
    }
    block_cmp(tot, sh);
    if (threadIdx.x == 0) {
        for (int j = 0; j < kCmp; ++j) scratch[kEnergyRecordOffset + j] = sh[j][0];
        *counter = 0u;
    }
}

template <typename RA>
cudaError_t compare_ref(const RA *a, const void *ref, bool ref_double, long long n, int nb, double *scratch,
                        cudaStream_t s) {
    if (ref_double)
        k_compare<RA, double><<<nb, kEnergyThreads, 0, s>>>(a, (const double *)ref, n, scratch);
    else
        k_compare<RA, float><<<nb, kEnergyThreads, 0, s>>>(a, (const float *)ref, n, scratch);
    return cudaGetLastError();
}

// Cooperative launch of kern (grid nb) when every block can be resident at once; clears the barrier
// word first.
template <typename K, typename... Args>
cudaError_t launch_cooperative(K kern, int nb, void *barrier, cudaStream_t s, Args... args) {
    int dev = 0, coop = 0, sms = 0, per_sm = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kEnergyThreads, 0);
    if (e != cudaSuccess) return e;
    if (!coop || (long long)per_sm * sms < nb) return cudaErrorNotSupported;
    // the barrier's arrival count and flag start at zero
    e = cudaMemsetAsync(barrier, 0, sizeof(unsigned long long), s);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(nb);
    cfg.blockDim = dim3(kEnergyThreads);
    cfg.dynamicSmemBytes = 0;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    const cudaError_t r = cudaLaunchKernelEx(&cfg, kern, args...);
    if (r == cudaErrorCooperativeLaunchTooLarge || r == cudaErrorNotSupported) {
        (void)cudaGetLastError();  // not launched: the caller runs one launch per step instead
        return cudaErrorNotSupported;
    }
    return r;
}

template <int NC, bool ENERGY>
cudaError_t steps_nc(const StepArgs &a, int nsteps, const CoefE &ke, double *scratch, double *records, unsigned polls,
                     cudaStream_t s) {
    // with ENERGY the partial sums' blocks and the reducing one
    const int nb = ENERGY ? energy_grid(a.g.sites) + 1 : (int)((a.g.sites + kEnergyThreads - 1) / kEnergyThreads);
    if (a.prec == LF2_F64)
        return launch_cooperative(k_steps<double, NC, 3, ENERGY, Coef64>, nb, scratch + kStepsBarrierWord, s, (double *)a.phi, (double *)a.phi_out,
                                  (double *)a.pi, a.comp, a.g, make_coef64(a.p, a.dt), ke, nsteps, scratch, records, polls);
    const Coef32 k = make_coef32(a.p, a.dt);
    if (a.prec == LF2_F32_KAHAN)
        return launch_cooperative(k_steps<float, NC, 1, ENERGY, Coef32>, nb, scratch + kStepsBarrierWord, s, (float *)a.phi, (float *)a.phi_out,
                                  (float *)a.pi, a.comp, a.g, k, ke, nsteps, scratch, records, polls);
    return launch_cooperative(k_steps<float, NC, 0, ENERGY, Coef32>, nb, scratch + kStepsBarrierWord, s, (float *)a.phi, (float *)a.phi_out,
                              (float *)a.pi, a.comp, a.g, k, ke, nsteps, scratch, records, polls);
}

template <bool ENERGY>
cudaError_t launch_steps(const StepArgs &a, int nsteps, double *scratch, double *records, bool no_wait, cudaStream_t s) {
    if (!a.drift || nsteps < 2) return cudaErrorNotSupported;
    // one site per thread; the launch itself checks that all blocks are resident
    if (a.g.sites > (ENERGY ? (long long)kStepsMaxBlocks * kEnergyThreads : steps_plain_max_sites()))
        return cudaErrorNotSupported;
    const CoefE ke = make_coefE(a.p);
    const unsigned polls = no_wait ? 0u : kBarrierPolls;
    switch (a.ncomp) {
        case 1: return steps_nc<1, ENERGY>(a, nsteps, ke, scratch, records, polls, s);
        case 2: return steps_nc<2, ENERGY>(a, nsteps, ke, scratch, records, polls, s);
        case 3: return steps_nc<3, ENERGY>(a, nsteps, ke, scratch, records, polls, s);
        case 4: return steps_nc<4, ENERGY>(a, nsteps, ke, scratch, records, polls, s);
        case 5: return steps_nc<5, ENERGY>(a, nsteps, ke, scratch, records, polls, s);
        case 6: return steps_nc<6, ENERGY>(a, nsteps, ke, scratch, records, polls, s);
        default: return cudaErrorNotSupported;
    }
}

}  // namespace

cudaError_t launch_steps_energy(const StepArgs &a, int nsteps, double *scratch, double *records, bool no_wait,
                                cudaStream_t s) {
    return launch_steps<true>(a, nsteps, scratch, records, no_wait, s);
}

long long steps_plain_max_sites() { return 8LL * device_sm_count() * kEnergyThreads; }

cudaError_t launch_steps_plain(const StepArgs &a, int nsteps, double *scratch, bool no_wait, cudaStream_t s) {
    return launch_steps<false>(a, nsteps, scratch, nullptr, no_wait, s);
}

cudaError_t steps_energy_timed_out(double *scratch, bool *out, cudaStream_t s) {
    unsigned long long word = 0;
    cudaError_t e = cudaMemcpyAsync(&word, scratch + kStepsStatusWord, sizeof word, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return e;
    *out = word != 0;
    if (*out) {
        e = cudaMemsetAsync(scratch + kStepsStatusWord, 0, sizeof word, s);  // reported once
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    }
    return e;
}

cudaError_t bounds_violations_energy(unsigned long long *n, bool reset) { return bounds_violations_here(n, reset); }

cudaError_t launch_compare(const void *a, bool a_double, const void *ref, bool ref_double, long long n,
                           double *scratch, cudaStream_t s) {
    const int nb = energy_grid(n);
    if (a_double) return compare_ref<double>((const double *)a, ref, ref_double, n, nb, scratch, s);
    return compare_ref<float>((const float *)a, ref, ref_double, n, nb, scratch, s);
}

cudaError_t launch_energy(const void *phi, const void *pi, const Geom &g, int ncomp, lf2_precision prec,
                          const lf2_params &p, double *scratch, double *record, cudaStream_t s) {
    const CoefE k = make_coefE(p);
    if (prec == LF2_F64) return launch_typed<double>(phi, pi, g, ncomp, k, scratch, record, s);
    return launch_typed<float>(phi, pi, g, ncomp, k, scratch, record, s);
}

cudaError_t launch_step_energy(const StepArgs &a, double *scratch, double *record, cudaStream_t s) {
    if (!a.drift) return cudaErrorInvalidValue;
    const CoefE ke = make_coefE(a.p);
    const int nb = energy_grid(a.g.sites);
    switch (a.ncomp) {
        case 1: step_energy_nc<1>(a, ke, nb, scratch, record, s); break;
        case 2: step_energy_nc<2>(a, ke, nb, scratch, record, s); break;
        case 3: step_energy_nc<3>(a, ke, nb, scratch, record, s); break;
        case 4: step_energy_nc<4>(a, ke, nb, scratch, record, s); break;
        case 5: step_energy_nc<5>(a, ke, nb, scratch, record, s); break;
        case 6: step_energy_nc<6>(a, ke, nb, scratch, record, s); break;
        default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

// ------------------------------------------------- fixed scratch for lf2_energy_noalloc
// Some callers cannot allocate device memory: code that runs while a memory pool or another
// framework owns the device allocator, or that must not make allocation calls at all.
// lf2_energy allocates its scratch on first use; lf2_energy_noalloc uses this file-scope array
// instead.  Every GPU that loads the library holds it until process exit.  Its size is fixed
// because the reduction grid has at most kEnergyBlocks blocks whatever the lattice: the
// partial rows, the record and the finished-block counter of any reduction fit, as the
// assertion below checks.  Static device memory starts zeroed; lf2_energy_noalloc also clears
// the counter before each launch.
static __device__ __align__(256) double g_energy_noalloc[kEnergyScratchDoubles];
static_assert(kEnergyRecordOffset >= kEnergyBlocks * kEnergySlots &&
                  kEnergyCounterOffset >= kEnergyRecordOffset + kEnergySlots &&
                  kEnergyCounterOffset + 1 <= kEnergyScratchDoubles,
              "the fixed scratch must hold kEnergyBlocks partial rows, the record and the counter");

namespace {
constexpr int kMaxDevices = 64;
std::mutex g_noalloc_mu;
double *g_noalloc_addr[kMaxDevices] = {};
}  // namespace

// The device address of g_energy_noalloc on the current device.  The first call on a device
// asks the runtime for it (host code cannot use the array's name as a device address) and
// caches it; later calls only read the cache.
cudaError_t energy_noalloc_scratch(double **out) {
    int dev = -1;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(g_noalloc_mu);
    if (!g_noalloc_addr[dev]) {
        void *addr = nullptr;
        e = cudaGetSymbolAddress(&addr, g_energy_noalloc);
        if (e != cudaSuccess) return e;
        g_noalloc_addr[dev] = static_cast<double *>(addr);
    }
    *out = g_noalloc_addr[dev];
    return cudaSuccess;
}

}  // namespace lf2
