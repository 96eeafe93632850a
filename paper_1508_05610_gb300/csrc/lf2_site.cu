// lf2_site.cu -- the shape-agnostic leapfrog kernels (any Nx, Ny, Nz): one thread per site, and a
// column walk for real FP32 fields; the first derivative; the precision conversions used by
// upload/download.
//
// In the per-site kernel each thread owns one site (x, y, z) of the row-major lattice and reads its
// six periodic neighbours x+-i (the Site jumps of Sec. 3.4 with the torus wrap of Sec. 3.3.1 done by
// index arithmetic instead of a stored halo).
#include <atomic>
#include <type_traits>

#include "lf2_bounds.cuh"
#include "lf2_internal.cuh"

namespace lf2 {
namespace {

constexpr int kThreads = 256;

// A site's NC components as accesses of the largest of 16, 8 and 4 bytes that divides them (field
// buffers are 16-byte aligned): whole sites of 2, 4 and 6 FP32 or 2 FP64 components take one to
// three vector accesses instead of one per component, each of which touched every line of the warp
// (133x121x112 FP32+Kahan step, k_site: 4 components 55.9 -> 31.4 us, 6 components 112 -> 51 us).
template <typename R, int BYTES>
struct Chunk;
template <>
struct Chunk<float, 4> {
    using T = float;
};
template <>
struct Chunk<float, 8> {
    using T = float2;
};
template <>
struct Chunk<float, 16> {
    using T = float4;
};
template <>
struct Chunk<double, 8> {
    using T = double;
};
template <>
struct Chunk<double, 16> {
    using T = double2;
};
template <typename R, int NC>
struct SiteChunks {
    static constexpr int BYTES = NC * (int)sizeof(R);
    static constexpr int CH = BYTES % 16 == 0 ? 16 : (BYTES % 8 == 0 ? 8 : 4);
    static constexpr int COUNT = BYTES / CH, E = CH / (int)sizeof(R);
    using V = typename Chunk<R, CH>::T;
};
template <typename R, int NC>
__device__ __forceinline__ void load_at(const R *__restrict__ p, R (&v)[NC]) {
    using C = SiteChunks<R, NC>;
#pragma unroll
    for (int q = 0; q < C::COUNT; ++q) {
        const typename C::V t = __ldg(reinterpret_cast<const typename C::V *>(p) + q);
        memcpy(&v[q * C::E], &t, C::CH);
    }
}
// Data the kernel also writes.  FP64 by L2 loads, which may be issued ahead of earlier stores (the
// punned pointers lose __restrict__; 257x193x161 complex FP64 runs 1.34 times as fast with them);
// FP32 by plain ones, since the chunks of a site share L1 lines (5 components: 1.1 times as fast).
template <typename R, int NC>
__device__ __forceinline__ void load_own(const R *p, R (&v)[NC]) {
    using C = SiteChunks<R, NC>;
    const typename C::V *c = reinterpret_cast<const typename C::V *>(p);
#pragma unroll
    for (int q = 0; q < C::COUNT; ++q) {
        const typename C::V t = sizeof(R) == 8 ? __ldcg(c + q) : c[q];
        memcpy(&v[q * C::E], &t, C::CH);
    }
}
template <typename R, int NC>
__device__ __forceinline__ void store_own(R *p, const R (&v)[NC]) {
    using C = SiteChunks<R, NC>;
#pragma unroll
    for (int q = 0; q < C::COUNT; ++q) {
        typename C::V t;
        memcpy(&t, &v[q * C::E], C::CH);
        reinterpret_cast<typename C::V *>(p)[q] = t;
    }
}

template <typename R, int NC>
__device__ __forceinline__ void load_site(const R *__restrict__ f, long long s, long long sites, R (&v)[NC]) {
    load_at<R, NC>(f + checked(s * NC, NC, sites * NC), v);
}

template <int NC>
__global__ void __launch_bounds__(kThreads) k_site_f64(const double *__restrict__ phi, double *__restrict__ phi_out,
                                                       double *__restrict__ pi, Geom g, Stride3 d, Coef64 k,
                                                       int drift) {
    for (SiteWalk w((long long)blockIdx.x * blockDim.x + threadIdx.x, g); w.s < g.sites; w.advance(d, g)) {
        const long long s = w.s;
        const int x = w.x, y = w.y, z = w.z;
        const long long row = (long long)g.nx;
        const long long plane = row * g.ny;
        double c[NC], xm[NC], xp[NC], ym[NC], yp[NC], zm[NC], zp[NC], p[NC], out[NC];
        const long long o = checked(s * NC, NC, g.sites * NC);
        load_site<double, NC>(phi, s, g.sites, c);
        load_site<double, NC>(phi, s - x + wrap_dn(x, g.nx), g.sites, xm);
        load_site<double, NC>(phi, s - x + wrap_up(x, g.nx), g.sites, xp);
        load_site<double, NC>(phi, s + (wrap_dn(y, g.ny) - y) * row, g.sites, ym);
        load_site<double, NC>(phi, s + (wrap_up(y, g.ny) - y) * row, g.sites, yp);
        load_site<double, NC>(phi, s + (wrap_dn(z, g.nz) - z) * plane, g.sites, zm);
        load_site<double, NC>(phi, s + (wrap_up(z, g.nz) - z) * plane, g.sites, zp);
        load_own<double, NC>(pi + o, p);
        update_f64<NC>(c, xm, xp, ym, yp, zm, zp, p, out, k);
        store_own<double, NC>(pi + o, p);
        if (drift) store_own<double, NC>(phi_out + o, out);
    }
}

// MODE 0: plain FP32 drift, 1: Kahan drift, 2: kick only.
template <int NC, int MODE>
__global__ void __launch_bounds__(kThreads) k_site_f32(const float *__restrict__ phi, float *__restrict__ phi_out,
                                                       float *__restrict__ pi, float *__restrict__ comp, Geom g,
                                                       Stride3 d, Coef32 k) {
    for (SiteWalk w((long long)blockIdx.x * blockDim.x + threadIdx.x, g); w.s < g.sites; w.advance(d, g)) {
        const long long s = w.s;
        const int x = w.x, y = w.y, z = w.z;
        const long long row = (long long)g.nx;
        const long long plane = row * g.ny;
        float c[NC], xm[NC], xp[NC], ym[NC], yp[NC], zm[NC], zp[NC], p[NC], cm[NC], out[NC];
        const long long o = checked(s * NC, NC, g.sites * NC);
        load_site<float, NC>(phi, s, g.sites, c);
        load_site<float, NC>(phi, s - x + wrap_dn(x, g.nx), g.sites, xm);
        load_site<float, NC>(phi, s - x + wrap_up(x, g.nx), g.sites, xp);
        load_site<float, NC>(phi, s + (wrap_dn(y, g.ny) - y) * row, g.sites, ym);
        load_site<float, NC>(phi, s + (wrap_up(y, g.ny) - y) * row, g.sites, yp);
        load_site<float, NC>(phi, s + (wrap_dn(z, g.nz) - z) * plane, g.sites, zm);
        load_site<float, NC>(phi, s + (wrap_up(z, g.nz) - z) * plane, g.sites, zp);
        load_own<float, NC>(pi + o, p);
        if constexpr (MODE == 2) {
            kick_f32<NC>(c, xm, xp, ym, yp, zm, zp, p, k);
            store_own<float, NC>(pi + o, p);
        } else {
            if (MODE == 1) load_own<float, NC>(comp + o, cm);
            update_f32<NC, MODE == 1>(c, xm, xp, ym, yp, zm, zp, p, cm, out, k);
            store_own<float, NC>(pi + o, p);
            store_own<float, NC>(phi_out + o, out);
            if (MODE == 1) store_own<float, NC>(comp + o, cm);
        }
    }
}

// One step of a real FP32 field on any lattice shape: a thread owns one (x, y) column of sites and
// walks a chunk of z-planes with planes z-1, z, z+1 of its column in registers; the x and y
// neighbours come from L1 and L2 (threads are numbered along the plane's rows, so a block's rows
// overlap).  Against k_site it has no index arithmetic per site and loads each column once
// instead of three times.  FP32+Kahan step, a plane at a time, 133x121x112: k_site 12.8 us, k_march 10.7 (14.8 before
// k_site's divisions went); 515x77x99: 21.6 and 17.9 us (27.2); 257x193x161: 47.6 and 46.7 (53.8).
// With 2 or more components k_site is as fast or faster (its vector accesses are aligned along the
// whole lattice), and in FP64 both wait for the FP64 pipe.
// Bound by the latency of the loads, so BATCH planes are loaded before the first is computed: two
// with the compensated drift, 257x193x161 45.4 -> 41.3 us, 521x509x301 385 -> 365, 515x77x99 17.3 ->
// 16.6 (in blocks of 512: 42.5, 371, 16.6; four planes: 52, 516, 20, too few warps for their
// registers), and chunks of at least two: 67x65x61 6.0 -> 4.1 us.  One with the plain drift, which has
// fewer loads (two: 26.5 -> 30 us at 257x193x161).
constexpr int kMarchThreads = 256;
constexpr int kMarchPlanes = 8;  // per chunk: two planes more to load than to compute; 4 to 32 within 5 %

template <bool KAHAN, int BATCH>
__global__ void __launch_bounds__(kMarchThreads) k_march(const float *__restrict__ phi, float *__restrict__ phi_out,
                                                         float *__restrict__ pi, float *__restrict__ comp, Geom g,
                                                         Coef32 k, int zchunk) {
    const int plane = g.nx * g.ny;
    const int i = blockIdx.x * kMarchThreads + threadIdx.x;
    if (i >= plane) return;
    const PlaneNbr n(i, g);
    const int z0 = blockIdx.y * zchunk, z1 = min(z0 + zchunk, g.nz);
    auto load = [&](long long at) { return __ldg(phi + checked(at, 1, g.sites)); };
    float below[1] = {load((long long)wrap_dn(z0, g.nz) * plane + i)}, cur[1] = {load((long long)z0 * plane + i)};
    for (int z = z0; z < z1; z += BATCH) {
        float next[BATCH], xm[BATCH][1], xp[BATCH][1], ym[BATCH][1], yp[BATCH][1], p[BATCH][1], cm[BATCH][1];
        long long at[BATCH];
#pragma unroll
        for (int b = 0; b < BATCH; ++b) {
            const int zb = min(z + b, z1 - 1);  // past the chunk: its last plane again, not used
            const long long pz = (long long)zb * plane;
            at[b] = checked(pz + i, 1, g.sites);
            next[b] = load((long long)wrap_up(zb, g.nz) * plane + i);
            xm[b][0] = load(pz + n.xm);
            xp[b][0] = load(pz + n.xp);
            ym[b][0] = load(pz + n.ym);
            yp[b][0] = load(pz + n.yp);
            p[b][0] = pi[at[b]];
            cm[b][0] = KAHAN ? comp[at[b]] : 0.0f;
        }
#pragma unroll
        for (int b = 0; b < BATCH; ++b) {
            if (z + b >= z1) break;
            float above[1] = {next[b]}, out[1];
            update_f32<1, KAHAN>(cur, xm[b], xp[b], ym[b], yp[b], below, above, p[b], cm[b], out, k);
            pi[at[b]] = p[b][0];
            phi_out[at[b]] = out[0];
            if (KAHAN) comp[at[b]] = cm[b][0];
            below[0] = cur[0];
            cur[0] = above[0];
        }
    }
}

int grid_for(long long sites) {
    long long b = (sites + kThreads - 1) / kThreads;
    const long long cap = 16LL * device_sm_count();
    if (b > cap) b = cap;
    if (b < 1) b = 1;
    return (int)b;
}

__global__ void k_from_f64_f32(const double *__restrict__ src, float *__restrict__ dst, long long n) {
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        dst[i] = (float)src[i];
}

__global__ void k_f32_to_f64(const float *__restrict__ src, double *__restrict__ dst, long long n) {
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        dst[i] = (double)src[i];
}

}  // namespace

cudaError_t bounds_violations_site(unsigned long long *n, bool reset) { return bounds_violations_here(n, reset); }

template <int NC>
void site_launch(const StepArgs &a, int grid, cudaStream_t s) {
    const Stride3 d = make_stride3((long long)grid * kThreads, a.g);
    if (a.prec == LF2_F64) {
        k_site_f64<NC><<<grid, kThreads, 0, s>>>((const double *)a.phi, (double *)a.phi_out, (double *)a.pi, a.g, d,
                                                 make_coef64(a.p, a.dt), a.drift ? 1 : 0);
        return;
    }
    const Coef32 k = make_coef32(a.p, a.dt);
    const float *phi = (const float *)a.phi;
    float *out = (float *)a.phi_out, *pi = (float *)a.pi;
    if (!a.drift)
        k_site_f32<NC, 2><<<grid, kThreads, 0, s>>>(phi, out, pi, a.comp, a.g, d, k);
    else if (a.prec == LF2_F32_KAHAN)
        k_site_f32<NC, 1><<<grid, kThreads, 0, s>>>(phi, out, pi, a.comp, a.g, d, k);
    else
        k_site_f32<NC, 0><<<grid, kThreads, 0, s>>>(phi, out, pi, a.comp, a.g, d, k);
}

cudaError_t launch_site_step(const StepArgs &a, cudaStream_t s) {
    if (a.g.sites == 0) return cudaSuccess;
    const int grid = grid_for(a.g.sites);
    switch (a.ncomp) {
        case 1: site_launch<1>(a, grid, s); break;
        case 2: site_launch<2>(a, grid, s); break;
        case 3: site_launch<3>(a, grid, s); break;
        case 4: site_launch<4>(a, grid, s); break;
        case 5: site_launch<5>(a, grid, s); break;
        case 6: site_launch<6>(a, grid, s); break;
        default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

cudaError_t launch_general_step(const StepArgs &a, cudaStream_t s) {
    const long long plane = (long long)a.g.nx * a.g.ny, bx = (plane + kMarchThreads - 1) / kMarchThreads;
    // chunks as long as they leave eight blocks per SM, and 16-bit grid and 32-bit plane indices
    const bool kahan = a.prec == LF2_F32_KAHAN;
    int zchunk = kMarchPlanes;
    while (zchunk > (kahan ? 2 : 1) && bx * ((a.g.nz + zchunk - 1) / zchunk) < 8LL * device_sm_count()) zchunk /= 2;
    const long long bz = (a.g.nz + zchunk - 1) / zchunk;
    if (a.g.sites == 0 || a.prec == LF2_F64 || a.ncomp != 1 || !a.drift || plane + kMarchThreads >= (1LL << 31) ||
        bz > 65535)
        return launch_site_step(a, s);
    const dim3 grid((unsigned)bx, (unsigned)bz);
    const Coef32 k = make_coef32(a.p, a.dt);
    const float *phi = (const float *)a.phi;
    float *out = (float *)a.phi_out, *pi = (float *)a.pi;
    if (kahan)
        k_march<true, 2><<<grid, kMarchThreads, 0, s>>>(phi, out, pi, a.comp, a.g, k, zchunk);
    else
        k_march<false, 1><<<grid, kMarchThreads, 0, s>>>(phi, out, pi, a.comp, a.g, k, zchunk);
    return cudaGetLastError();
}

// ------------------------------------------------------------ symmetric difference
namespace {

// Any row length: a thread per element of the grid stride, so that neighbouring threads read
// neighbouring elements whatever the dimension.  g: the lattice in units of `inner` elements (1, and
// the row nx * ncomp units with x-neighbours `dist` = ncomp units apart; for rows of 2^31 elements and
// more in sites, with inner = ncomp and dist = 1); the coordinates advance by additions.  Bound by
// latency: the loads of kDerivBatch<R> elements are issued together (one at a time kept 10 KB per SM
// in flight, 1.5 TB/s): 257x193x161, the three dimensions, 3 components FP32 386 -> 231 us, FP64
// (two elements; four leave small lattices with a ragged last round) 410 -> 347 us.
template <typename R>
constexpr int kDerivBatch = sizeof(R) == 8 ? 2 : 4;

template <typename R>
__global__ void __launch_bounds__(kThreads) k_derivative(const R *__restrict__ src, R *__restrict__ dst, Geom g,
                                                         Stride3 d, int inner, int dist, int dim, R inv2dx) {
    const long long row = g.nx, plane = row * g.ny;
    SiteWalk w((long long)blockIdx.x * blockDim.x + threadIdx.x, g);
    while (w.s < g.sites) {
        const long long s0 = w.s;
        long long up[kDerivBatch<R>], dn[kDerivBatch<R>];
        int n = 0;
#pragma unroll
        for (int u = 0; u < kDerivBatch<R>; ++u) {
            up[u] = dn[u] = s0;  // past the end: an element of the lattice, not used
            if (w.s >= g.sites) continue;
            if (dim == 0) {
                up[u] = w.s + (w.x >= g.nx - dist ? dist - row : dist);
                dn[u] = w.s + (w.x < dist ? row - dist : -dist);
            } else if (dim == 1) {
                up[u] = w.s + (wrap_up(w.y, g.ny) - w.y) * row;
                dn[u] = w.s + (wrap_dn(w.y, g.ny) - w.y) * row;
            } else {
                up[u] = w.s + (wrap_up(w.z, g.nz) - w.z) * plane;
                dn[u] = w.s + (wrap_dn(w.z, g.nz) - w.z) * plane;
            }
            ++n;
            w.advance(d, g);
        }
        for (int a = 0; a < inner; ++a) {
            R hi[kDerivBatch<R>], lo[kDerivBatch<R>];
#pragma unroll
            for (int u = 0; u < kDerivBatch<R>; ++u) {
                hi[u] = __ldg(src + up[u] * inner + a);
                lo[u] = __ldg(src + dn[u] * inner + a);
            }
#pragma unroll
            for (int u = 0; u < kDerivBatch<R>; ++u)
                if (u < n) dst[(s0 + u * d.sites) * inner + a] = (hi[u] - lo[u]) * inv2dx;
        }
    }
}

// Rows made of whole 16-byte vectors: a thread takes one vector (E elements) of kDerivRows rows of a
// plane, all loads before the first use.  Bound: HBM, one read and one write of the field.  Along y
// and z the two neighbours are vectors of other rows.  Along x they are NC elements away: within the
// thread's vector or in the adjacent lane's (warp shuffle; the first lane of a warp and the last of
// a row load theirs) for the component counts of at most E (DIM 0), single loads from L1 otherwise
// (DIM 3).  256^3, the three dimensions together: 3 components FP32 390 -> 191 us (one, two, four
// rows per thread: 195, 191, 201), 1 component 113 -> 70, 6 components 740 -> 368; FP64 is bound by
// its subtraction and product on the FP64 pipe (3 components 662 -> 591).
constexpr int kDerivRows = 2;

template <typename R, int NC, int DIM>
__global__ void __launch_bounds__(256) k_derivative_rows(const R *__restrict__ src, R *__restrict__ dst, Geom g,
                                                         int ncomp, R inv2dx) {
    constexpr int E = 16 / sizeof(R);
    static_assert(NC <= E, "the x-neighbours of a vector lie in the vectors next to it");
    using V = typename std::conditional<sizeof(R) == 8, double2, float4>::type;
    const long long rowE = (long long)g.nx * ncomp, planeE = rowE * g.ny;
    const int y0 = blockIdx.y * kDerivRows, z = blockIdx.z;
    const long long e0 = ((long long)blockIdx.x * blockDim.x + threadIdx.x) * E;
    const bool active = e0 < rowE;
    R up[kDerivRows][E], dn[kDerivRows][E];
#pragma unroll
    for (int r = 0; r < kDerivRows; ++r) {
        const int y = y0 + r;
        const bool on = active && y < g.ny;  // y is the same for the whole block
        const long long base = (long long)z * planeE + (long long)y * rowE;
        if constexpr (DIM == 0) {
            R v[E];
            V t{};
            if (on) t = __ldg(reinterpret_cast<const V *>(src + base + e0));
            memcpy(v, &t, 16);
            R left[NC], right[NC];
            const int lane = threadIdx.x & 31;
#pragma unroll
            for (int a = 0; a < NC; ++a) {
                left[a] = __shfl_up_sync(0xffffffffu, v[E - NC + a], 1);
                right[a] = __shfl_down_sync(0xffffffffu, v[a], 1);
            }
            if (on && lane == 0) {
#pragma unroll
                for (int a = 0; a < NC; ++a) {
                    const long long e = e0 - NC + a;
                    left[a] = __ldg(src + base + (e < 0 ? e + rowE : e));
                }
            }
            if (on && (lane == 31 || e0 + E >= rowE)) {
#pragma unroll
                for (int a = 0; a < NC; ++a) {
                    const long long e = e0 + E + a;
                    right[a] = __ldg(src + base + (e >= rowE ? e - rowE : e));
                }
            }
#pragma unroll
            for (int j = 0; j < E; ++j) {
                dn[r][j] = j < NC ? left[j] : v[j < NC ? 0 : j - NC];
                up[r][j] = j + NC < E ? v[j + NC < E ? j + NC : 0] : right[j + NC < E ? 0 : j + NC - E];
            }
        } else if constexpr (DIM == 3) {
#pragma unroll
            for (int j = 0; j < E; ++j) {
                const long long u = e0 + j + ncomp, d = e0 + j - ncomp;
                up[r][j] = on ? __ldg(src + base + (u >= rowE ? u - rowE : u)) : R(0);
                dn[r][j] = on ? __ldg(src + base + (d < 0 ? d + rowE : d)) : R(0);
            }
        } else if (on) {
            const long long du = DIM == 1 ? (long long)(wrap_up(y, g.ny) - y) * rowE : (long long)(wrap_up(z, g.nz) - z) * planeE;
            const long long dd = DIM == 1 ? (long long)(wrap_dn(y, g.ny) - y) * rowE : (long long)(wrap_dn(z, g.nz) - z) * planeE;
            const V a = __ldg(reinterpret_cast<const V *>(src + base + du + e0));
            const V b = __ldg(reinterpret_cast<const V *>(src + base + dd + e0));
            memcpy(up[r], &a, 16);
            memcpy(dn[r], &b, 16);
        }
    }
#pragma unroll
    for (int r = 0; r < kDerivRows; ++r) {
        if (!active || y0 + r >= g.ny) continue;
        R out[E];
#pragma unroll
        for (int j = 0; j < E; ++j) out[j] = (up[r][j] - dn[r][j]) * inv2dx;
        V o;
        memcpy(&o, out, 16);
        __stcs(reinterpret_cast<V *>(dst + (long long)z * planeE + (long long)(y0 + r) * rowE + e0), o);
    }
}

template <typename R>
cudaError_t launch_rows(const void *src, void *dst, const Geom &g, int ncomp, int dim, R inv2dx, cudaStream_t s) {
    constexpr int E = 16 / (int)sizeof(R);
    const long long vecs = (long long)g.nx * ncomp / E;
    // whole warps of about equal blocks along a row, at most 256 threads (192 vectors: 192 threads)
    const long long nb = (vecs + 255) / 256;
    const int threads = (int)(((vecs + nb - 1) / nb + 31) / 32 * 32);
    const dim3 grid((unsigned)((vecs + threads - 1) / threads), (unsigned)((g.ny + kDerivRows - 1) / kDerivRows), g.nz);
    const R *a = (const R *)src;
    R *d = (R *)dst;
    if (dim == 1)
        k_derivative_rows<R, 1, 1><<<grid, threads, 0, s>>>(a, d, g, ncomp, inv2dx);
    else if (dim == 2)
        k_derivative_rows<R, 1, 2><<<grid, threads, 0, s>>>(a, d, g, ncomp, inv2dx);
    else if (ncomp == 1)
        k_derivative_rows<R, 1, 0><<<grid, threads, 0, s>>>(a, d, g, ncomp, inv2dx);
    else if (ncomp == 2)
        k_derivative_rows<R, 2, 0><<<grid, threads, 0, s>>>(a, d, g, ncomp, inv2dx);
    else if (ncomp == 3 && E >= 3)
        k_derivative_rows<R, E < 3 ? 1 : 3, 0><<<grid, threads, 0, s>>>(a, d, g, ncomp, inv2dx);
    else if (ncomp == 4 && E >= 4)
        k_derivative_rows<R, E < 4 ? 1 : 4, 0><<<grid, threads, 0, s>>>(a, d, g, ncomp, inv2dx);
    else
        k_derivative_rows<R, 1, 3><<<grid, threads, 0, s>>>(a, d, g, ncomp, inv2dx);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_derivative(const void *src, void *dst, const Geom &g, int ncomp, lf2_precision prec, int dim,
                              double dx, cudaStream_t s) {
    if (g.sites == 0) return cudaSuccess;
    const int esz = prec == LF2_F64 ? 8 : 4;
    const bool rows_ok = ((long long)g.nx * ncomp * esz) % 16 == 0 && ((uintptr_t)src | (uintptr_t)dst) % 16 == 0 &&
                         g.ny <= 65535 && g.nz <= 65535;
    if (rows_ok) {
        return prec == LF2_F64 ? launch_rows<double>(src, dst, g, ncomp, dim, 0.5 / dx, s)
                               : launch_rows<float>(src, dst, g, ncomp, dim, (float)(0.5 / dx), s);
    }
    const bool elements = (long long)g.nx * ncomp < (1LL << 31);
    const int inner = elements ? 1 : ncomp, dist = elements ? ncomp : 1;
    const Geom u = elements ? Geom{g.nx * ncomp, g.ny, g.nz, g.sites * ncomp} : g;
    const int grid = grid_for(u.sites);
    const Stride3 d = make_stride3((long long)grid * kThreads, u);
    if (prec == LF2_F64)
        k_derivative<double><<<grid, kThreads, 0, s>>>((const double *)src, (double *)dst, u, d, inner, dist, dim, 0.5 / dx);
    else
        k_derivative<float><<<grid, kThreads, 0, s>>>((const float *)src, (float *)dst, u, d, inner, dist, dim,
                                                      (float)(0.5 / dx));
    return cudaGetLastError();
}

cudaError_t launch_convert_from_f64(const double *src, void *dst, long long n, lf2_precision prec, cudaStream_t s) {
    if (n == 0) return cudaSuccess;
    if (prec == LF2_F64) return cudaMemcpyAsync(dst, src, (size_t)n * sizeof(double), cudaMemcpyDeviceToDevice, s);
    k_from_f64_f32<<<grid_for(n), kThreads, 0, s>>>(src, (float *)dst, n);
    return cudaGetLastError();
}

cudaError_t launch_convert_to_f64(const void *src, double *dst, long long n, lf2_precision prec, cudaStream_t s) {
    if (n == 0) return cudaSuccess;
    if (prec == LF2_F64) return cudaMemcpyAsync(dst, src, (size_t)n * sizeof(double), cudaMemcpyDeviceToDevice, s);
    k_f32_to_f64<<<grid_for(n), kThreads, 0, s>>>((const float *)src, dst, n);
    return cudaGetLastError();
}

int device_sm_count() {
    // one entry per device ordinal; concurrent first calls store the same value
    static std::atomic<int> cache[64];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 152;
    int n = cache[dev].load(std::memory_order_relaxed);
    if (n > 0) return n;
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n < 1) {
        (void)cudaGetLastError();
        return 152;
    }
    cache[dev].store(n, std::memory_order_relaxed);
    return n;
}

}  // namespace lf2
