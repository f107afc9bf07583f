// Internal declarations shared by the library's translation units.
#pragma once

#include <cuda_runtime.h>

#include <atomic>
#include <string>
#include <vector>

#include "../../include/aem_rjsmc.h"

namespace aem {

constexpr double kPi = 3.14159265358979323846;
constexpr double kMu0 = 4e-7 * kPi;
constexpr int kTab64Turn = 1024, kTab64Octave = 256;  // entries of the FP64 forward kernel's tables (d_tab64)

// Records the message returned by aem_last_error() and passes the code through.
int fail(int code, const std::string &msg);
int cuda_fail(cudaError_t err, const char *what);

#define AEM_CUDA_TRY(expr)                                        \
    do {                                                          \
        cudaError_t _e = (expr);                                  \
        if (_e != cudaSuccess) return ::aem::cuda_fail(_e, #expr); \
    } while (0)

// How many CTAs of a kernel fit an SM with that much dynamic shared memory:
// asked of the runtime once and kept in *slot (0: not asked yet), with the
// kernel's dynamic shared memory limit raised to all that its static share
// leaves (the same value whoever asks, so no caller lowers it under another)
// and the SM's unified storage given to shared memory.  Setting both and asking
// on every launch cost 6 us.
template <class Kernel>
int resident_ctas(std::atomic<int> *slot, Kernel kern, int threads, size_t smem, int device, int *out) {
    int n = slot->load(std::memory_order_relaxed);
    if (n == 0) {
        cudaFuncAttributes fa{};
        int optin = 0;
        AEM_CUDA_TRY(cudaFuncGetAttributes(&fa, kern));
        AEM_CUDA_TRY(cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, device));
        AEM_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                          optin - (int)fa.sharedSizeBytes));
        AEM_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout,
                                          (int)cudaSharedmemCarveoutMaxShared));
        AEM_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kern, threads, smem));
        if (n > 0) slot->store(n, std::memory_order_relaxed);
    }
    *out = n;
    return AEM_OK;
}

// Host-side tables (double) and their device copies (float and double).
struct SystemTables {
    double a = 0, h = 0, current = 1;
    int F = 0, G = 0, K = 0, cc_form = 0;
    std::vector<double> freqs, omega, times, lam, hw, T;  // T is G x F
};

// Gates (and log-likelihood) from spectra [P][F] by the transform of the
// given aem_gates_mode; y_obs rows advance every obs_per models (gates_tc.cu).
int gates_from_spectrum(const aem_system *sys, const float *imh, int P, int mode, const double *y_obs,
                        int obs_per, const double *eps_an, double eps_mn, float *gates, double *ll,
                        cudaStream_t stream);
}  // namespace aem

struct aem_system {
    aem::SystemTables host;
    int device = 0;
    // device tables: omega[F], lam[K], hw[K], T[G*F] in both precisions
    float *d_omega_f = nullptr, *d_lam_f = nullptr, *d_hw_f = nullptr, *d_T_f = nullptr;
    // the FP32 forward kernel's length unit (a power of two, metres) and its
    // abscissae in it
    float len = 1.f, *d_lamu_f = nullptr;
    // float pairs (value, what its rounding left): omega mu0 in that unit [F];
    // T [F*G] (by frequency), then a bound on each gate's sum of |T| over |Im H| <= 1 [G]
    float2 *d_wmu_f = nullptr, *d_T_pair = nullptr;
    // the FP64 forward kernel's tables: sine and cosine of 2 pi j / kTab64Turn in
    // pairs, then 2^(j / kTab64Octave)
    double *d_tab64 = nullptr;
    double *d_omega_d = nullptr, *d_lam_d = nullptr, *d_hw_d = nullptr, *d_T_d = nullptr;
    int num_sms = 0;
    // device status word: kernels record AEM_ERR_TIMEOUT here when a bounded
    // wait gives up (read and cleared by aem_system_status)
    int *d_status = nullptr;
    // diagnostics of the bounded waits (aem_debug_bounded_wait): their iteration limit (0: the
    // default) and whether the tensor-core transform's CTAs issue nothing for their first tile
    unsigned int wait_spins = 0;
    int wait_skip_mma = 0;
    // launch shape of the FP32 forward kernel per lmax (index into its shape
    // table, -1 = none recorded), set by aem_autotune_forward / aem_forward_shape
    int f32_shape[AEM_MAX_LAYERS + 1];
    aem_system() {
        for (int &s : f32_shape) s = -1;
    }
    // CTAs per SM of each kernel, asked once (resident_ctas): the FP32 forward
    // shapes and the adjoint per lmax, the tensor-core transform per mode
    mutable std::atomic<int> fwd_ctas[AEM_F32_SHAPES + 2][AEM_MAX_LAYERS + 1] = {};
    mutable std::atomic<int> grad_ctas[AEM_MAX_LAYERS + 1] = {};
    mutable std::atomic<int> tc_ctas[3] = {};
    // the FP32 forward kernel's depth cutoff (aem_system_set_depth_cutoff):
    // attenuation exponent, 0 = the whole stack always
    float depth_att = 20.f;
};

namespace aem {
// Builds the Hankel rule and the transform matrix on the host (system.cpp).
int build_tables(const aem_system_desc *desc, SystemTables *out);
// FP32 forward + log-likelihood where consecutive blocks of
// models_per_sounding models use consecutive rows of y_obs (forward.cu).
// counter: optional device int the dynamic-scheduled shapes use for model
// claiming instead of a per-launch stream-ordered allocation.  active:
// optional device int; when it holds 0 the launch does nothing (a sweep of a
// captured stage loop that the device-side sweep count switched off).  valid:
// optional per-model device flags; a model whose flag is 0 is skipped and its
// ll left as it was (a proposal that was no move, which the accept step
// ignores).
int loglik_f32_soundings(const aem_system *sys, const aem_models_f32 *models, const double *y_obs,
                         int models_per_sounding, const double *eps_an, double eps_mn, double *ll,
                         cudaStream_t stream, int *counter = nullptr, const int *active = nullptr,
                         const int8_t *valid = nullptr);
// The plain FP64 forward model + log-likelihood with the same per-sounding
// rows of y_obs (forward.cu); active and valid as above.
int loglik_f64_soundings(const aem_system *sys, const aem_models_f64 *models, const double *y_obs,
                         int models_per_sounding, const double *eps_an, double eps_mn, double *ll,
                         cudaStream_t stream, const int *active = nullptr, const int8_t *valid = nullptr);
// Gates [P][G] and log-likelihood (may be NULL) of the FP32 forward kernel
// with per-sounding rows of y_obs (forward.cu); counter and valid as above.
int loglik_gates_f32_soundings(const aem_system *sys, const aem_models_f32 *models, const double *y_obs,
                               int models_per_sounding, const double *eps_an, double eps_mn, double *ll, float *gates,
                               cudaStream_t stream, int *counter = nullptr, const int8_t *valid = nullptr);
// Log-likelihood and its merged-layer gradient [P][lmax][5] with the same
// per-sounding rows of y_obs (adjoint.cu).  work: optional device scratch of
// grad_work_bytes(P, G) bytes (the claim counters and the gates); without it
// the call takes stream-ordered scratch of that size for its duration.  With
// it the call makes no allocation, so it can be captured inside a
// conditional graph body.  valid: optional per-model device flags; a model
// whose flag is 0 is skipped (its ll and gradient left as they were).
size_t grad_work_bytes(int n_models, int G);
int loglik_grad_f32_soundings(const aem_system *sys, const aem_models_f32 *models, const double *y_obs,
                              int models_per_sounding, const double *eps_an, double eps_mn, double *ll, float *grad,
                              cudaStream_t stream, void *work = nullptr, const int8_t *valid = nullptr);
// Gates (and log-likelihood) from spectra [P][F] by the transform of the
// given aem_gates_mode; y_obs rows advance every obs_per models (gates_tc.cu).
int gates_from_spectrum(const aem_system *sys, const float *imh, int P, int mode, const double *y_obs,
                        int obs_per, const double *eps_an, double eps_mn, float *gates, double *ll,
                        cudaStream_t stream);
}  // namespace aem
