// lf2_spectrum.cu -- binned power spectrum of one field component, or of all components
// summed (a diagnostic; the paper's PlanFFT role, Sec. 3.6, for cubic lattices as there).
//
// P(k) = |phi~(k)|^2 / V with phi~(k) = sum_x phi(x) exp(-i k.x), k_i = 2 pi m_i / (N dx).
// Mode (m_x, m_y, m_z) goes to shell b = floor(sqrt(m_x^2 + m_y^2 + m_z^2)), an exact integer
// square root, so the shell of every mode is the same whatever the rounding of |k|.  The
// transform is cuFFT's real-to-complex FFT (a library call); the half spectrum it returns
// stands for each mode k != -k twice.  The binning kernel accumulates (power, |k|, count) per
// shell in a per-block shared histogram, writes one row per block, and a second kernel sums
// the rows in a fixed order.  Shared-memory accumulation order varies between runs, so results
// are reproducible to FP64 rounding, not bitwise.
#include <cuda_runtime.h>
#include <cufft.h>

#include <cmath>
#include <cstring>
#include <new>
#include <vector>

#include "lf2_handles.h"

using namespace lf2;

namespace {

constexpr int kBinThreads = 256;
constexpr int kMaxBins = 1024;

template <typename R>
__global__ void k_extract(const R *__restrict__ f, R *__restrict__ out, long long sites, int ncomp, int comp) {
    for (long long s = (long long)blockIdx.x * blockDim.x + threadIdx.x; s < sites; s += (long long)gridDim.x * blockDim.x)
        out[s] = f[s * ncomp + comp];
}

// The largest x >= 0 with x^2 <= v, exactly.
__device__ __forceinline__ int floor_sqrt(long long v) {
    long long x = (long long)sqrtf((float)v);
    while (x * x > v) --x;
    while ((x + 1) * (x + 1) <= v) ++x;
    return (int)x;
}

__device__ __forceinline__ void add_mode(double2 c, double &acc) { acc = __fma_rn(c.y, c.y, __fma_rn(c.x, c.x, acc)); }
__device__ __forceinline__ void add_mode(float2 c, double &acc) {
    const double re = widen(c.x), im = widen(c.y);
    acc = __fma_rn(im, im, __fma_rn(re, re, acc));
}

// Sums of the modes of each shell.  The rows (ky, kz), (+-ky, +-kz) and with ky and kz exchanged, up
// to eight, have the same |k| at every kx, so a warp adds the modes of all of them, lane for kx,
// before it looks at shells: one square root and one shell per eight modes, and eight independent
// coalesced loads in flight.  Along kx the shells are runs of neighbouring lanes, which are summed
// by shuffles, so that the block's histogram in shared memory gets one addition per shell and warp.
// 256^3 FP32: 75 us, against 438 us with an atomic for each of power, |k| and count per mode.
// Bound: the FP64 pipe (two products per mode, then the square roots).
// add_power: add this component's power to the rows a previous component's binning wrote,
// leaving the |k| sums and mode counts (the same for every component) as they are.
template <typename C>
__global__ void __launch_bounds__(kBinThreads) k_bin(const C *__restrict__ spec, int n, int nbins, double kunit,
                                                     double inv_volume, double *__restrict__ partials, int add_power) {
    extern __shared__ double hist[];  // nbins powers, nbins |k| sums, nbins counts (64-bit integers)
    unsigned long long *cnt = reinterpret_cast<unsigned long long *>(hist + 2 * nbins);
    for (int i = threadIdx.x; i < 2 * nbins; i += kBinThreads) hist[i] = 0.0;
    for (int i = threadIdx.x; i < nbins; i += kBinThreads) cnt[i] = 0ull;
    __syncthreads();
    const int hx = n / 2 + 1, half = n / 2, lane = threadIdx.x & 31;
    const bool even = n % 2 == 0;
    const double both = 2.0 * inv_volume;
    auto self = [&](int k) { return k == 0 || (even && k == half); };  // its own mirror image
    const long long pairs = (long long)hx * (hx + 1) / 2;  // 0 <= ky <= kz <= half
    const int segs = (hx + 31) / 32;
    const long long items = pairs * segs;
    const long long warp0 = ((long long)blockIdx.x * kBinThreads + threadIdx.x) / 32;
    for (long long it = warp0; it < items; it += (long long)gridDim.x * (kBinThreads / 32)) {
        const long long p = it / segs;
        const int x = (int)(it - p * segs) * 32 + lane;
        // p = kz (kz + 1) / 2 + ky
        int kz = (floor_sqrt(8 * p + 1) - 1) / 2;
        const int ky = (int)(p - (long long)kz * (kz + 1) / 2);
        const long long q = (long long)ky * ky + (long long)kz * kz;
        if (floor_sqrt(q) >= nbins) continue;  // the whole row lies beyond the shells asked for
        C v[8];
        bool have[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            have[j] = !((j & 1) && self(ky)) && !((j & 2) && self(kz)) && !((j & 4) && ky == kz);
            const int a = (j & 1) ? n - ky : ky, b = (j & 2) ? n - kz : kz;
            const long long row = (j & 4) ? (long long)a * n + b : (long long)b * n + a;
            if (have[j] && x < hx) v[j] = __ldg(spec + row * hx + x);
        }
        const long long s2 = q + (long long)x * x;
        const int shell = x < hx ? floor_sqrt(s2) : 0x7fffffff;
        const bool in = shell < nbins;
        double power = 0.0, ksum = 0.0;
        int images = 0;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            if (!have[j]) continue;  // the same for the whole warp
            ++images;
            if (in) add_mode(v[j], power);
        }
        unsigned count = 0u;
        if (in) {
            const int w = self(x) ? 1 : 2;  // kx and -kx
            power *= w == 1 ? inv_volume : both;  // before the shell's sum, which could overflow where its mean does not
            count = (unsigned)(w * images);
            if (!add_power) ksum = (double)count * sqrt((double)s2);
        }
        // sums over runs of equal shells, left in the run's first lane
        for (int off = 1; off < 32; off *= 2) {
            const int other = __shfl_down_sync(0xffffffffu, shell, off);
            const bool same = lane + off < 32 && other == shell;
            if (!__any_sync(0xffffffffu, same)) break;  // no run is longer
            const double dp = __shfl_down_sync(0xffffffffu, power, off), dk = __shfl_down_sync(0xffffffffu, ksum, off);
            const unsigned dc = __shfl_down_sync(0xffffffffu, count, off);
            if (same) {
                power += dp;
                ksum += dk;
                count += dc;
            }
        }
        const int before = __shfl_up_sync(0xffffffffu, shell, 1);
        if (in && (lane == 0 || before != shell)) {
            atomicAdd(&hist[shell], power);
            if (!add_power) {
                atomicAdd(&hist[nbins + shell], ksum);
                atomicAdd(&cnt[shell], (unsigned long long)count);
            }
        }
    }
    __syncthreads();
    double *out = partials + (size_t)blockIdx.x * 3 * nbins;
    for (int i = threadIdx.x; i < nbins; i += kBinThreads) {
        if (add_power) {
            out[i] += hist[i];
        } else {
            out[i] = hist[i];
            out[nbins + i] = hist[nbins + i] * kunit;
            out[2 * nbins + i] = (double)cnt[i];
        }
    }
}

// A warp per sum over the blocks' rows: lanes in steps of 32 rows, then pairwise (a fixed order).
__global__ void __launch_bounds__(kBinThreads) k_bin_final(const double *__restrict__ partials, int nblocks, int nbins,
                                                           double *__restrict__ out) {
    const int i = (blockIdx.x * kBinThreads + threadIdx.x) / 32, lane = threadIdx.x % 32;
    if (i >= 3 * nbins) return;
    double s = 0.0;
    for (int b = lane; b < nblocks; b += 32) s += partials[(size_t)b * 3 * nbins + i];
    for (int w = 16; w > 0; w >>= 1) s += __shfl_down_sync(0xffffffffu, s, w);
    if (lane == 0) out[i] = s;
}

// The lattice keeps its plans: making one took over half of a 256^3 call.
constexpr size_t kIdleFftPlans = 2;

lf2_status take_plan(lf2_lattice lat, bool dbl, FftPlan *out) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return cuda_error(e, "cudaGetDevice");
    {
        std::lock_guard<std::mutex> lock(lat->fft_mu);
        for (size_t i = 0; i < lat->fft_idle.size(); ++i) {
            if (lat->fft_idle[i].device != dev || lat->fft_idle[i].dbl != dbl) continue;
            *out = lat->fft_idle[i];
            lat->fft_idle.erase(lat->fft_idle.begin() + i);
            return LF2_OK;
        }
    }
    const int n = lat->n[0];
    cufftHandle h = 0;
    size_t work = 0;
    cufftResult r = cufftCreate(&h);
    if (r != CUFFT_SUCCESS)
        return set_error(r == CUFFT_ALLOC_FAILED ? LF2_ERR_NOMEM : LF2_ERR_CUDA, "cuFFT error %d", (int)r);
    r = cufftSetAutoAllocation(h, 0);
    if (r == CUFFT_SUCCESS) r = cufftMakePlan3d(h, n, n, n, dbl ? CUFFT_D2Z : CUFFT_R2C, &work);
    if (r != CUFFT_SUCCESS) {
        cufftDestroy(h);
        return set_error(r == CUFFT_ALLOC_FAILED ? LF2_ERR_NOMEM : LF2_ERR_CUDA, "cuFFT error %d", (int)r);
    }
    *out = FftPlan{dev, dbl, (int)h, work};
    return LF2_OK;
}

// Keeps a plan whose work is done, unless the call failed or enough are kept.
void give_plan(lf2_lattice lat, const FftPlan &p, bool good) {
    if (good) {
        std::lock_guard<std::mutex> lock(lat->fft_mu);
        if (lat->fft_idle.size() < kIdleFftPlans) {
            try {
                lat->fft_idle.push_back(p);
                return;
            } catch (const std::bad_alloc &) {
            }
        }
    }
    cufftDestroy((cufftHandle)p.handle);
}

}  // namespace

namespace lf2 {
void release_fft_plans(lf2_lattice lat) {
    for (const FftPlan &p : lat->fft_idle) cufftDestroy((cufftHandle)p.handle);
    lat->fft_idle.clear();
}
}  // namespace lf2

extern "C" lf2_status lf2_power_spectrum(lf2_field f, int comp, int nbins, double dx, double *power, double *kmean,
                                         double *count, void *stream) {
    if (!f || !power || !kmean || !count) return set_error(LF2_ERR_INVALID, "NULL argument");
    const int *n3 = f->lat->n;
    if (n3[0] != n3[1] || n3[1] != n3[2])
        return set_error(LF2_ERR_UNSUPPORTED, "the power spectrum needs a cubic lattice (as the paper's FFT)");
    if (comp < -1 || comp >= f->ncomp) return set_error(LF2_ERR_INVALID, "component %d out of range", comp);
    if (nbins < 1 || nbins > kMaxBins) return set_error(LF2_ERR_INVALID, "nbins must be 1 to %d", kMaxBins);
    if (!(dx > 0.0)) return set_error(LF2_ERR_INVALID, "dx must be > 0");
    const int n = n3[0];
    const long long sites = f->lat->sites;
    const bool dbl = f->prec == LF2_F64;
    const size_t rsz = dbl ? sizeof(double) : sizeof(float);
    const size_t csz = 2 * rsz;
    cudaStream_t s = (cudaStream_t)stream;
    const int kBinBlocks = 4 * device_sm_count();  // four histogram blocks per SM
    FftPlan plan{};
    lf2_status st = take_plan(f->lat, dbl, &plan);
    if (st != LF2_OK) return st;
    // one allocation: a component's values (a one-component field is read where it is), its half
    // spectrum, the transform's work area, the partial rows and the sums
    auto aligned = [](size_t b) { return (b + 255) / 256 * 256; };
    const bool copy = f->ncomp > 1;
    const size_t real_b = copy ? aligned((size_t)sites * rsz) : 0, spec_b = aligned((size_t)n * n * (n / 2 + 1) * csz),
                 work_b = aligned(plan.work_bytes), part_b = aligned((size_t)kBinBlocks * 3 * nbins * sizeof(double)),
                 out_b = (size_t)3 * nbins * sizeof(double);
    char *arena = nullptr;
    cudaError_t e = cudaMalloc(&arena, real_b + spec_b + work_b + part_b + out_b);
    if (e != cudaSuccess) st = cuda_error(e, "spectrum buffers");
    void *real = arena, *spec = arena + real_b, *work = arena + real_b + spec_b;
    double *partials = (double *)(arena + real_b + spec_b + work_b), *out = partials + part_b / sizeof(double);
    if (st == LF2_OK) {
        cufftResult r = cufftSetStream(plan.handle, s);
        if (r == CUFFT_SUCCESS) r = cufftSetWorkArea(plan.handle, work);
        if (r != CUFFT_SUCCESS) st = set_error(LF2_ERR_CUDA, "cuFFT error %d", (int)r);
    }
    // one component, or every component in order with their powers added bin by bin
    const int c0 = comp < 0 ? 0 : comp, c1 = comp < 0 ? f->ncomp : comp + 1;
    const double kunit = 2.0 * M_PI / (n * dx);
    const double inv_volume = 1.0 / ((double)n * n * n);
    const size_t smem = (size_t)3 * nbins * sizeof(double);
    for (int c = c0; c < c1 && st == LF2_OK; ++c) {
        const long long cap = 16LL * device_sm_count();
        const int g = (int)((sites + 255) / 256 < cap ? (sites + 255) / 256 : cap);
        if (!copy)
            real = f->val[f->front];
        else if (dbl)
            k_extract<double><<<g, 256, 0, s>>>((const double *)f->val[f->front], (double *)real, sites, f->ncomp, c);
        else
            k_extract<float><<<g, 256, 0, s>>>((const float *)f->val[f->front], (float *)real, sites, f->ncomp, c);
        e = cudaGetLastError();
        if (e != cudaSuccess) {
            st = cuda_error(e, "component copy");
            break;
        }
        const cufftResult r = dbl ? cufftExecD2Z(plan.handle, (cufftDoubleReal *)real, (cufftDoubleComplex *)spec)
                                  : cufftExecR2C(plan.handle, (cufftReal *)real, (cufftComplex *)spec);
        if (r != CUFFT_SUCCESS) {
            st = set_error(LF2_ERR_CUDA, "cuFFT error %d", (int)r);
            break;
        }
        const int add = c > c0;
        if (dbl)
            k_bin<double2><<<kBinBlocks, kBinThreads, smem, s>>>((const double2 *)spec, n, nbins, kunit, inv_volume, partials, add);
        else
            k_bin<float2><<<kBinBlocks, kBinThreads, smem, s>>>((const float2 *)spec, n, nbins, kunit, inv_volume, partials, add);
        e = cudaGetLastError();
        if (e != cudaSuccess) st = cuda_error(e, "binning");
    }
    if (st == LF2_OK) {
        k_bin_final<<<(3 * nbins * 32 + kBinThreads - 1) / kBinThreads, kBinThreads, 0, s>>>(partials, kBinBlocks, nbins, out);
        e = cudaGetLastError();
        double host[3 * kMaxBins];
        if (e == cudaSuccess) e = cudaMemcpyAsync(host, out, out_b, cudaMemcpyDeviceToHost, s);
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);
        if (e != cudaSuccess) st = cuda_error(e, "binning");
        if (st == LF2_OK) {
            memcpy(power, host, nbins * sizeof(double));
            memcpy(kmean, host + nbins, nbins * sizeof(double));
            memcpy(count, host + 2 * nbins, nbins * sizeof(double));
        }
    }
    give_plan(f->lat, plan, st == LF2_OK);
    if (arena) cudaFree(arena);
    if (st != LF2_OK) return st;
    for (int b = 0; b < nbins; ++b) {  // sums -> means
        if (count[b] > 0) {
            power[b] /= count[b];
            kmean[b] /= count[b];
        }
    }
    return LF2_OK;
}
