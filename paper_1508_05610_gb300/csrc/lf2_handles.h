// lf2_handles.h -- host-side definitions of the opaque handles of the C ABI (lattice, field,
// ensemble) and small helpers shared by the API, tuner and ensemble sources.
#pragma once

#include <atomic>
#include <mutex>
#include <string>
#include <vector>

#include "lf2_internal.cuh"

// A cuFFT plan of a lattice without its work area (lf2_spectrum.cu).
struct FftPlan {
    int device;
    bool dbl;
    int handle;        // cufftHandle
    size_t work_bytes;
};

struct lf2_lattice_s {
    int dim;
    int n[3];
    int halo;
    long long sites;
    std::atomic<int> users{0};  // fields and ensembles still attached
    // FFT plans not in use, at most kIdleFftPlans: a call takes one out (or makes one) and gives it
    // back when its stream is done, so threads never share a plan; destroyed with the lattice
    std::mutex fft_mu;
    std::vector<FftPlan> fft_idle;
};

struct lf2_field_s {
    lf2_lattice lat = nullptr;
    int ncomp = 0;
    lf2_precision prec = LF2_F64;
    size_t esize = 0;  // bytes per stored element
    long long count = 0;  // sites * ncomp
    void *val[2] = {nullptr, nullptr};  // value buffers; val[front] is current
    bool own_val[2] = {false, false};
    int front = 0;
    float *comp[2] = {nullptr, nullptr};  // Kahan compensation of phi (F32_KAHAN); comp[cfront] current
    bool own_comp[2] = {false, false};
    int cfront = 0;
    double *energy_scratch = nullptr;  // kFieldScratchDoubles: partial rows, record, counter, multi-step rows (device)
    double *energy_host = nullptr;     // one pinned lf2_energy_t
    lf2_ensemble ensemble = nullptr;   // the ensemble this field is a member of, if any
};

namespace lf2 {

// Sets the calling thread's last-error message and returns `s`.
lf2_status set_error(lf2_status s, const char *fmt, ...) __attribute__((format(printf, 2, 3)));
lf2_status cuda_error(cudaError_t e, const char *what);

// Host-side switches (lf2_api.cu): LF2_FAULT=<what> injects a failure; LF2_TUNE picks how
// lf2_leapfrog uses tuned plans.
bool fault_injected(const char *what);
enum class TuneMode { Off, On, Force };
TuneMode tune_mode();

// Field helpers (lf2_api.cu).
lf2_status ensure_dynamic(lf2_field phi, cudaStream_t s);               // phi back buffer (+ compensation)
lf2_status ensure_tblock(lf2_field phi, lf2_field pi, cudaStream_t s);  // + pi and compensation back buffers
StepArgs step_args(lf2_field phi, lf2_field pi, const lf2_params *p, double dt, bool drift);
TbArgs tb_args(lf2_field phi, lf2_field pi, const lf2_params *p);

// nsteps of lf2_leapfrog_ex with checked arguments; LF2_KERNEL_AUTO is the untuned choice, whatever plan
// the shape has.
lf2_status leapfrog_run(lf2_field phi, lf2_field pi, const lf2_params *p, int nsteps, const lf2_step_config *cfg,
                        cudaStream_t s);

// Energy scratch of a field, which the multi-step runs use too (lf2_api.cu).
lf2_status ensure_energy_scratch(lf2_field f);

// Tuned kernel plan for a lattice shape (filled by lf2_tune); false if none.
bool plan_lookup(const int n[3], int ncomp, lf2_precision prec, lf2_step_config *out);

// Destroys the lattice's idle FFT plans (lf2_spectrum.cu).
void release_fft_plans(lf2_lattice lat);

inline Geom geom_of(const lf2_lattice_s *lat) { return Geom{lat->n[0], lat->n[1], lat->n[2], lat->sites}; }

}  // namespace lf2
