// Internal declarations shared by the FDAS CUDA translation units (not part of the C ABI).
#pragma once

#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include "../../include/fdas.h"

namespace fdas {

// The last CUDA error met on this thread (fdas_last_error): note() records e with the function and
// line that met it and returns e unchanged; fail() turns e into a status, recording it unless the
// record already holds the same error from a deeper call.
cudaError_t note(cudaError_t e, const char *where, int line);
fdas_status fail(cudaError_t e, const char *where, int line);
#define FDAS_NOTE(e) ::fdas::note((e), __func__, __LINE__)
#define FDAS_STATUS(e) ::fdas::fail((e), __func__, __LINE__)

// Derived sizes of one parameter set.
struct Geometry {
    int n_temp;   // template rows
    int c;        // centre row (zero drift), (n_temp-1)/2
    int n_tap;    // taps per template
    int h;        // half width, (n_tap-1)/2
    int fft_len;  // overlap-save segment length F
    int keep;     // valid outputs per segment, L = F - n_tap + 1
    int precision;  // FDAS_FP32, FDAS_BF16X3 or FDAS_FP16S
};

inline Geometry geometry(const fdas_params &p) {
    Geometry g;
    g.n_temp = p.n_temp;
    g.c = (p.n_temp - 1) / 2;
    g.n_tap = p.n_tap;
    g.h = (p.n_tap - 1) / 2;
    g.fft_len = p.fft_len;
    g.keep = p.fft_len - p.n_tap + 1;
    g.precision = p.precision;
    return g;
}

// Workspace layout of the harmonic-sum stage (all 8-byte words):
//   [0, n_harm)                 raw crossing counters (low 32 bits used)
//   [n_harm, 2 n_harm)          peak keys, one per plane
//   [4 n_harm, 4 n_harm + n_harm*FDAS_RAW_CAP)  raw candidate keys, FDAS_RAW_CAP per plane
struct HsWorkspace {
    unsigned long long *counters;
    unsigned long long *peaks;
    unsigned long long *raw;
};

inline HsWorkspace hs_workspace(void *ws, int n_harm) {
    unsigned long long *w = static_cast<unsigned long long *>(ws);
    return HsWorkspace{w, w + n_harm, w + 4 * n_harm};
}

inline size_t hs_workspace_words(int n_harm) { return (size_t)n_harm * (FDAS_RAW_CAP + 4); }

// Largest batch: the per-spectrum tables travel as kernel parameters (a few KB to 20 KB).
constexpr int kMaxBatch = FDAS_MAX_BATCH;

// One spectrum of a batch, as the batched convolution kernel reads it.
struct ConvJob {
    const float2 *spec;
    float *plane;
    unsigned long long ld;
    int n;
    int seg0;  // first segment of this spectrum in the batch
    // This spectrum's harmonic-sum workspace (HsWorkspace), for HP_1 taken in the convolution.
    unsigned long long *counters;
    unsigned long long *peaks;
    unsigned long long *raw;
};
struct ConvBatch {
    int count;
    int total_segments;
    ConvJob job[kMaxBatch];
};

// One spectrum of a batch, as the batched harmonic-sum kernels read it.
struct HsJob {
    const float *plane;
    unsigned long long ld;
    int n;
    int jend;   // fundamental columns of this spectrum in the harmonic sum (harmonic_units)
    int unit0;  // first unit of this spectrum in the launch
    unsigned long long *counters;  // this spectrum's workspace (HsWorkspace)
    unsigned long long *peaks;
    unsigned long long *raw;
    fdas_cand *cands;
    uint32_t *counts;
    fdas_cand *peak_out;
};
struct HsBatch {
    int count;
    int units;  // of all spectra
    int cols;   // columns per unit
    HsJob job[kMaxBatch];
};

// Launches that overlap the end of the kernel before them on the stream (programmatic dependent launch).
// Such a kernel's CTAs may start once every CTA of the kernel before has called pdl_trigger() or has
// ended; pdl_wait() returns when that kernel has completed and its writes are visible. Both are no-ops in a plain
// launch. What keeps this safe:
//   - Only kernels that follow one of the same call are launched this way (`chained`).
//   - A thread calls pdl_wait() before it reads what an earlier kernel of the call writes and before it writes
//     anything, and some thread of every such kernel does call it, so completion still goes down the chain: a kernel
//     that has completed has waited for the one before it. (A CTA that finds no work may end without.)
//   - Before the wait a kernel reads the call's inputs at most: the convolution with HP_1 loads the spectrum, the
//     template bank and the thresholds while the reset runs. That is safe because the reset in front of it is a
//     plain launch, behind everything that was on the stream before the call. Do not chain that reset.
//   - None reads through L1, before the wait, what a kernel still running may write (the convolution's look back
//     at its own outputs goes to L2).
// Only the reset of the workspace triggers early. Elsewhere the launch alone is worth it: a search takes
// 36.6 -> 30.8 us at 4099 bins, 516.6 -> 510.5 us at 2^21. With a trigger in the convolution, CTAs of
// the harmonic sum sat on SMs whose memory was still split for the convolution's shared buffers, and had
// next to no L1 for their gathers: 585 us at 2^21 bins.
#ifdef __CUDACC__
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;\n" ::: "memory"); }
template <class... P, class... A>
cudaError_t launch_pdl(bool chained, void (*kernel)(P...), dim3 grid, int threads, size_t smem, cudaStream_t s,
                       A &&...args) {
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = chained ? 1 : 0;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, P(args)...);
}
#endif

// Kernel launchers (each returns cudaGetLastError() of its launch).
cudaError_t launch_templates(const fdas_params &p, void *d_tmpl, cudaStream_t s);
// Convolution launch for g.precision: the FP32 kernel or the tensor-core kernel.
cudaError_t launch_convolve(const Geometry &g, const float2 *spec, size_t n, const float2 *tmpl, float *plane,
                            size_t ld, int ctas_per_sm, int templates_per_item, cudaStream_t s);
cudaError_t launch_convolve_fp32(const Geometry &g, const float2 *spec, size_t n, const float2 *tmpl,
                                 float *plane, size_t ld, int ctas_per_sm, int templates_per_item, cudaStream_t s);
// Segments of a spectrum of n bins.
int segment_count(const Geometry &g, size_t n);
// SMs of the current device.
cudaError_t sm_count(int *sms);
// Tensor-core form: one CTA per SM (all of Tensor Memory).
constexpr int kTcMaxCtasPerSm = 1;
// With ws also HP_1, as launch_convolve_hp1; a batch always takes it.
cudaError_t launch_convolve_tc(const Geometry &g, const float2 *spec, size_t n, const float2 *tmpl, float *plane,
                               size_t ld, int ctas_per_sm, int templates_per_item, cudaStream_t s,
                               const float *thresh = nullptr, unsigned harm_mask = 0u, const HsWorkspace *ws = nullptr);
cudaError_t prepare_convolve_batch_tc();
cudaError_t launch_convolve_batch_tc(const Geometry &g, const ConvBatch &batch, const float2 *tmpl,
                                     int templates_per_item, int sms, const float *thresh, unsigned harm_mask,
                                     cudaStream_t s);
cudaError_t device_status_tc(unsigned *flags, bool clear);
cudaError_t device_status_tc_async(unsigned *h_flags, cudaStream_t s);
// Resident CTAs per SM of the convolution kernel for g.precision.
inline int convolve_ctas_per_sm(const Geometry &g) { return g.precision == FDAS_FP32 ? 3 : kTcMaxCtasPerSm; }
// Zeroes the harmonic-sum workspace's counters and peak keys. Never chained in front of a convolution (launch_pdl).
cudaError_t launch_hs_reset(const fdas_params &p, const HsWorkspace &ws, cudaStream_t s, bool chained = false);
// Convolution for g.precision that also emits the HP_1 candidates (threshold thresh[0..n_temp), when bit 0 of
// harm_mask is set) and the HP_1 peak into the workspace, which a plain launch of this call has just reset.
cudaError_t launch_convolve_hp1(const Geometry &g, const float2 *spec, size_t n, const float2 *tmpl, float *plane,
                                size_t ld, const float *thresh, unsigned harm_mask, const HsWorkspace &ws,
                                cudaStream_t s);
// Status bits set by kernels on the device (bit 0: a bounded wait timed out); optionally cleared.
cudaError_t device_status(unsigned *flags, bool clear);
// Enqueues on s copies of the two translation units' status words into h_flags2[0] and h_flags2[1]
// (valid once s reaches them; with pageable host memory the call itself waits for that).
cudaError_t device_status_async(unsigned *h_flags2, cudaStream_t s);
// Sets the status word to flags (the tensor-core unit's word is cleared).
cudaError_t set_device_status(unsigned flags);
// FP32 FFMA-chain throughput of the current device over about ms milliseconds (diag.cu).
cudaError_t measure_fp32_peak(float ms, double *tflops, float *elapsed_ms);
// Runs a kernel whose bounded wait must give up; returns the status bits it left (then cleared).
cudaError_t check_wait_timeout(unsigned *flags);
cudaError_t prepare_convolve_batch();
// Batched convolution: one launch over every segment of every spectrum, at most ctas_per_sm CTAs per SM. It takes every
// spectrum's HP_1 into its workspace (ConvJob counters / peaks / raw, reset beforehand).
cudaError_t launch_convolve_batch_hp1(const Geometry &g, const ConvBatch &batch, const float2 *tmpl, int ctas_per_sm,
                                      int templates_per_item, int sms, const float *thresh, unsigned harm_mask,
                                      cudaStream_t s);
// Harmonic sum. With hp1_done the workspace was reset before the convolution, which already took
// HP_1. chained: the kernel before on the stream is this call's convolution.
cudaError_t launch_harmonic(const fdas_params &p, const float *plane, size_t n, size_t ld,
                            const float *thresh, fdas_cand *cands, uint32_t *counts, fdas_cand *peaks,
                            const HsWorkspace &ws, cudaStream_t s, bool hp1_done = false, bool chained = false);
// The sums and their detection with FDAS_INDEX_HIGHEST (workspace reset beforehand).
cudaError_t launch_hs_highest(const fdas_params &p, const float *plane, size_t n, size_t ld, const float *thresh,
                              const HsWorkspace &ws, int sms, cudaStream_t s);
// The driver's id of the current device's context (made current if it is not), unique for the life
// of the process: caches keyed by it never hand out a resource of a context that cudaDeviceReset
// destroyed.
cudaError_t current_context_id(unsigned long long *id);
// Whether `device` has a live primary context.
bool primary_context_active(int device);
// Batched harmonic sum: the columns per unit for these spectra; the units of one spectrum and its
// columns jend; the launch (reset unless hp1_done, sum, finalize).
int harmonic_columns(const fdas_params &p, const size_t *lengths, int count, bool hp1_done, int sms);
int harmonic_units(const fdas_params &p, size_t n, int cols, bool hp1_done, int *jend);
cudaError_t prepare_harmonic_batch();
cudaError_t launch_harmonic_batch(const fdas_params &p, const HsBatch &batch, const float *thresh, cudaStream_t s,
                                  bool hp1_done = false);
// Zeroes every spectrum's counters and peak keys.
cudaError_t launch_hs_reset_batch(const fdas_params &p, const HsBatch &batch, cudaStream_t s);

}  // namespace fdas
