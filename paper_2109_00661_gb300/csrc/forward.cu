// Batched forward model and Gaussian log-likelihood on sm_103a.
//
// One CTA (FP32; grid-stride over models) or cluster of CTAs (FP64; by
// frequency) works on one model at a time.  For that model it stages, in shared
// memory, s_n(w_f) = i w_f mu0 sigma_n(w_f) for every frequency node and merged
// layer (Cole-Cole, Section 2), then its threads sweep the flattened (frequency,
// Hankel abscissa) index space.  Each item runs the bottom-up TE reflection
// recursion over the layers (the hot loop: F*K*L layer-steps per model) and
// weights Im R_0 by the folded Hankel weight; the sums over the abscissae of a
// frequency are taken in a fixed order from a per-item value buffer.  The FP32
// kernel also drops the layers under its depth cutoff (depth_cutoff.h).  The
// epilogue applies the G x F step-off transform and, for
// the likelihood entry points, the Gaussian log-likelihood of Section 2.3.2
// (gates in float pairs, FP32 terms and an FP64 sum in the FP32 kernel, FP64
// throughout in the FP64 one).
//
// Recursion used (quasi-static TE mode, exp(+i w t)):
//   u_n = sqrt(lambda^2 + s_n), Re u_n > 0
//   r   = (u_n - u_{n+1}) / (u_n + u_{n+1})
//   R_n = (r + R_{n+1} E) / (1 + r R_{n+1} E),  E = exp(-2 u_{n+1} h_{n+1})
// carried projectively as R = N / D so the Moebius step needs no division:
//   N' = r D + N E,  D' = D + r N E.  |D| grows by at most 2x per layer.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <cstdint>
#include <type_traits>

#include "aem_internal.h"
#include "depth_cutoff.h"
#include "f32x2.h"
#include "te_roots.h"

namespace aem {
namespace {

constexpr unsigned kFull = 0xffffffffu;

template <class R>
__device__ __forceinline__ R warp_sum(R v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
    return v;
}

template <class R>
struct ModelsView {
    int n, lmax;
    const int8_t *nlayers;
    const R *logsig, *logh, *m, *logtau, *c;
};

// ===================================================================== FP64
// The plain double-precision form.  This part retires about 1.65 FP64
// operations a clock per SM (1/78 of FP32), so the kernel's time is its count
// of FP64 operations, and everything else is free: roots and reciprocals take
// the hardware's 20-bit estimates and one third-order step, the exponential and
// the sine and cosine a table in shared memory and a short polynomial, signs,
// exponents and table indices integer instructions.  61 FP64 operations per
// layer-step (154 with the library's sqrt, rsqrt, division, exp and sincos):
// 1,024 models of 1..10 layers, 60 frequencies, 200 abscissae, 19.4 -> 7.71 ms,
// at the rate the FP64 pipe allows.
//
// The recursion is the FP32 kernel's, (N, D) <- (r D + N E, D + r N E) in w =
// sqrt(2) u with the interface coefficient from the roots and their moduli.
// Carrying the field (e = D + P, h = w (D - P)) in place of r takes 53
// operations (7.0 ms), but e and h then keep the phase of the layers below,
// which Im R_0 has to cancel even where the layers above hide them: an error of
// 2^-53 times the conductivity contrast, 3e-12 of the spectrum on layers of
// 1e-4 and 1 S/m under a small loop near the ground and 1e-7 at a contrast of
// 1e16.  Here it is 5e-16 and 1e-14, on all stacks tried no more than with
// the library's functions and the differenced s.
namespace f64 {

constexpr int kExN = kTab64Octave, kScN = kTab64Turn;
constexpr double kShift = 6755399441055744.0;  // 1.5 * 2^52: the low word of x + kShift is round(x)

// Tables of the complex exponential (Tang 1989's scheme): 2^(j / kExN), sine
// and cosine of 2 pi j / kScN (kTab64Doubles in this order, f64_tables in system.cpp).
struct Tables {
    double2 sc[kScN];
    double ex[kExN];
};

// Per layer: -sqrt(2) h, and it in the tables' steps (times kExN / ln 2 and
// kScN / (2 pi)).
struct Thick {
    double h, he, hp;
};

// E = exp(-sqrt(2) h w).  With k the nearest step, the fused x h' - k is the
// exact remainder f, |f| <= 1/2; e^(f ln2 / 256) - 1 to f^4 (the next term is
// 4e-17), sin and cos of f pi / 512 to f^5 and f^4 (5e-22, 1e-18).
__device__ __forceinline__ void exp_c(double wre, double wim, const Thick &t, const Tables *tab, double &Ex,
                                      double &Ey) {
    constexpr double a = 0.69314718055994530942 / kExN, b = 6.28318530717958647693 / kScN;
    const double n = fma(t.he, wre, kShift);
    const int k = __double2loint(n);
    const double f = fma(t.he, wre, kShift - n);
    double q = fma(f, a * a * a * a / 24.0, a * a * a / 6.0);
    q = fma(q, f, a * a / 2.0);
    q = fma(q, f, a);
    const double T = tab->ex[k & (kExN - 1)];
    double e = fma(q * f, T, T);
    e = __hiloint2double(__double2hiint(e) + (int)((unsigned)(k >> 8) << 20), __double2loint(e));
    // below exp(-700): the steps themselves, from n's bits (a NaN of either sign
    // stays, and so does a thickness of infinity: exp(-inf) (cos, sin)(-inf))
    constexpr long long kGone = 0x4338000000000000ll - 258530;
    const bool gone = __double_as_longlong(n) < kGone && (unsigned)__double2hiint(n) < 0xfff00000u;
    const double m = fma(t.hp, wim, kShift);
    double sn, cs;
    if ((unsigned)(__double2hiint(m) - 0x43380000 + 0x20000) < 0x40000u) {  // |steps| < 2^49
        const double g = fma(t.hp, wim, kShift - m), g2 = g * g;
        double p = fma(g2, b * b * b * b * b / 120.0, -b * b * b / 6.0);
        p = fma(p, g2, b);
        const double sr = p * g;
        const double cr = fma(g2, b * b * b * b / 24.0, -b * b / 2.0) * g2;  // cos - 1
        const double2 v = tab->sc[__double2loint(m) & (kScN - 1)];
        sn = fma(v.y, sr, fma(v.x, cr, v.x));
        cs = fma(-v.x, sr, fma(v.y, cr, v.y));
    } else {
        sincos(t.h * wim, &sn, &cs);
    }
    Ex = gone ? 0.0 : e * cs;
    Ey = gone ? 0.0 : e * sn;
}

struct Rec {  // per frequency and layer
    double sx, sy, sy2;
};
struct C {
    double x, y;
};
struct Root {  // w = sqrt(2 (lambda^2 + s)) and m = |w|^2 / 2
    double x, y, m;
};

// w = sqrt(2 (x + i y)).  From the 20-bit estimate y of 1 / sqrt(v), g = v y and
// e = 1 - g y: sqrt(v) = g (1 + c) and 1 / sqrt(v) = y (1 + c) with c = e (1/2 +
// 3/8 e), up to 5/16 e^3 < 2^-55.
__device__ __forceinline__ double rsq_est(double v) {
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(v));
    return y;
}
__device__ __forceinline__ Root root(double lam2, const Rec &s) {
    const double x = lam2 + s.sx;
    const double v = fma(x, x, s.sy2);
    const double y1 = rsq_est(v), g1 = v * y1, e1 = fma(-g1, y1, 1.0);
    const double m = fma(e1 * fma(e1, 0.375, 0.5), g1, g1);
    const double t = m + fabs(x);
    const double y2 = rsq_est(t), g2 = t * y2, e2 = fma(-g2, y2, 1.0);
    const double c = e2 * fma(e2, 0.375, 0.5);
    const double p = fma(c, g2, g2), o = s.sy * fma(c, y2, y2);
    const bool pos = __double2hiint(x) >= 0;
    return {pos ? p : o, pos ? o : p, m};
}
__device__ __forceinline__ double rcp(double v) {
    double y;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(v));
    const double r = fma(-v, y, 1.0);  // 1 / v = y (1 + r + r^2 + ..)
    return fma(fma(r, r, r), y, y);
}
// The interface coefficient between a (above) and b from the roots and their
// moduli (the form of te_roots.h), and that of the air above the top layer, whose
// root is the real wair and modulus lam2.
__device__ __forceinline__ C rcoef(const Root &a, const Root &b) {
    const double i = rcp(fma(a.y, b.y, fma(a.x, b.x, a.m + b.m)));
    return {(a.m - b.m) * i, fma(a.y, b.x, -(a.x * b.y)) * i};
}
__device__ __forceinline__ C rcoef_air(double lam2, double wair, const Root &b) {
    const double i = rcp(fma(wair, b.x, lam2 + b.m));
    return {(lam2 - b.m) * i, -(wair * b.y) * i};
}

// Im R_0 of one (lambda, frequency); rec: the frequency's layers.
__device__ __forceinline__ double im_r0(double lam2, double wair, const Rec *__restrict__ rec,
                                        const Thick *__restrict__ th, int L, const Tables *tab) {
    Root b = root(lam2, rec[L - 1]);
    if (L == 1) return rcoef_air(lam2, wair, b).y;
    Root a = root(lam2, rec[L - 2]);
    C N = rcoef(a, b), D = {1.0, 0.0};
#pragma unroll 1
    for (int n = L - 2;; --n) {
        double Ex, Ey;
        exp_c(a.x, a.y, th[n], tab, Ex, Ey);
        C r;
        if (n > 0) {
            b = a;
            a = root(lam2, rec[n - 1]);
            r = rcoef(a, b);
        } else {
            r = rcoef_air(lam2, wair, a);
        }
        const C P = {fma(N.x, Ex, -(N.y * Ey)), fma(N.x, Ey, N.y * Ex)};
        N = {fma(r.x, D.x, fma(-r.y, D.y, P.x)), fma(r.x, D.y, fma(r.y, D.x, P.y))};
        D = {fma(r.x, P.x, fma(-r.y, P.y, D.x)), fma(r.x, P.y, fma(r.y, P.x, D.y))};
        if (n == 0) break;
    }
    return fma(N.y, D.x, -(N.x * D.y)) * rcp(fma(D.x, D.x, D.y * D.y));
}

}  // namespace f64

constexpr int kThreads64 = 256;
constexpr int kChunk64 = 8;  // frequencies whose items share the value buffer
constexpr int kTab64Doubles = (int)(sizeof(f64::Tables) / sizeof(double));
static_assert(kTab64Doubles == 2 * kTab64Turn + kTab64Octave && kTab64Octave == 256, "");

// Shared memory (dynamic): vals [kChunk64 * K], lam2 [K], wair [K], hw [K],
// rec [kChunk64 * lmax], imh [F].
size_t smem_bytes_f64(int F, int K, int lmax) {
    return sizeof(double) * ((size_t)kChunk64 * K + 3 * (size_t)K + F) + sizeof(f64::Rec) * (size_t)kChunk64 * lmax;
}

// A cluster of C CTAs per model, CTA r over the r-th of C equal ranges of the
// frequencies, a chunk at a time: layer records, items (one per thread and
// pass, into the value buffer), one fixed-order sum per frequency.  Rank 0
// collects the spectrum through distributed shared memory and forms gates and
// likelihood.
__global__ void __launch_bounds__(kThreads64) forward_f64_kernel(ModelsView<double> mv, int F, int G, int K,
                                                               int cc_form, const double *__restrict__ g_omega,
                                                               const double *__restrict__ g_lam,
                                                               const double *__restrict__ g_hw,
                                                               const double *__restrict__ g_T,
                                                               const double *__restrict__ g_tab,
                                                               double *__restrict__ gates_out,
                                                               double *__restrict__ imh_out,
                                                               const double *__restrict__ y_obs, int obs_per,
                                                               const double *__restrict__ eps_an, double eps_mn,
                                                               double *__restrict__ ll_out,
                                                               const int *__restrict__ active,
                                                               const int8_t *__restrict__ valid) {
    namespace cg = cooperative_groups;
    cg::cluster_group cl = cg::this_cluster();
    const int C = (int)cl.num_blocks(), rank = (int)cl.block_rank();
    const int p = blockIdx.x / C;
    if (active && *active == 0) return;  // a gated launch the caller switched off on the device
    if (valid && !valid[p]) return;      // a proposal the caller will not use (the whole cluster)
    extern __shared__ __align__(16) unsigned char smem_raw[];
    double *vals = reinterpret_cast<double *>(smem_raw);
    double *lam2 = vals + (size_t)kChunk64 * K, *wair = lam2 + K, *hw = wair + K, *imh = hw + K;
    f64::Rec *rec = reinterpret_cast<f64::Rec *>(imh + F);
    __shared__ f64::Tables tab;
    __shared__ double lsig[AEM_MAX_LAYERS], lm[AEM_MAX_LAYERS], ltau[AEM_MAX_LAYERS], lc[AEM_MAX_LAYERS];
    __shared__ f64::Thick th[AEM_MAX_LAYERS];
    __shared__ double ll_part[2];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int L = mv.nlayers[p];
    for (int j = tid; j < kTab64Doubles; j += kThreads64) reinterpret_cast<double *>(&tab)[j] = g_tab[j];
    for (int k = tid; k < K; k += kThreads64) {
        const double l = g_lam[k];
        lam2[k] = l * l;
        wair[k] = 1.4142135623730951 * l;
        hw[k] = g_hw[k];
    }
    if (tid < L) {
        const size_t o = (size_t)p * mv.lmax + tid;
        lsig[tid] = exp10(mv.logsig[o]);
        const double h = -1.4142135623730951 * exp10(mv.logh[o]);
        th[tid] = {h, h * (f64::kExN / 0.69314718055994530942), h * (f64::kScN / 6.28318530717958647693)};
        lm[tid] = mv.m[o];
        ltau[tid] = exp10(mv.logtau[o]);
        lc[tid] = mv.c[o];
    }
    const int f0 = F * rank / C, f1 = F * (rank + 1) / C;
    for (int fc = f0; fc < f1; fc += kChunk64) {
        const int nf = min(kChunk64, f1 - fc);
        __syncthreads();
        // Cole-Cole per (frequency, layer): x = (w tau)^c e^{i pi c / 2}, s = i w mu0 sigma
        for (int i = tid; i < nf * L; i += kThreads64) {
            const int f = i / L, n = i - f * L;
            const double w = g_omega[fc + f];
            const double sig = lsig[n], mm = lm[n];
            double sr = sig, si = 0.0;
            if (mm != 0.0) {
                const double cc = lc[n];
                const double mag = exp(cc * log(w * ltau[n]));
                double sp, cp;
                sincospi(0.5 * cc, &sp, &cp);
                const double xr = 1.0 + mag * cp, xi = mag * sp;  // 1 + x
                const double den = xr * xr + xi * xi;
                // every form is written without cancellation (see the FP32 kernel)
                if (cc_form == AEM_CC_PAPER) {
                    // sigma_inf ((1 - m) + x) / (1 + x)
                    sr = sig * (((1.0 - mm) + mag * cp) * xr + xi * xi) / den;
                    si = sig * (mm * xi / den);
                } else if (cc_form == AEM_CC_LITERAL) {
                    // sigma_0 (1 + (1 - m) x) / (1 + x)
                    const double br = 1.0 + (1.0 - mm) * mag * cp, bi = (1.0 - mm) * mag * sp;
                    sr = sig * (br * xr + bi * xi) / den;
                    si = -sig * (mm * xi / den);
                } else {
                    // sigma_0 (1 + x) / (1 + (1 - m) x)
                    const double br = 1.0 + (1.0 - mm) * mag * cp, bi = (1.0 - mm) * mag * sp;
                    const double bd = br * br + bi * bi;
                    sr = sig * (xr * br + xi * bi) / bd;
                    si = sig * (mm * xi / bd);
                }
            }
            const double sx = -w * kMu0 * si, sy = w * kMu0 * sr;
            rec[f * L + n] = {sx, sy, sy * sy};
        }
        __syncthreads();
        int f = tid / K, k = tid - f * K;
        for (int item = tid; item < nf * K; item += kThreads64) {
            vals[item] = hw[k] * f64::im_r0(lam2[k], wair[k], rec + f * L, th, L, &tab);
            k += kThreads64;
            while (k >= K) {
                k -= K;
                ++f;
            }
        }
        __syncthreads();
        // a warp per frequency: lanes stride its values, then a shuffle tree
        for (int j = warp; j < nf; j += kThreads64 / 32) {
            double acc = 0.0;
            for (int q = lane; q < K; q += 32) acc += vals[j * K + q];
            acc = warp_sum<double>(acc);
            if (lane == 0) imh[fc + j] = acc;
        }
    }
    if (C > 1) {
        cl.sync();
        if (rank == 0)
            for (int j = f1 + tid; j < F; j += kThreads64) {
                int r = (int)((long long)j * C / F);
                while (r + 1 < C && F * (r + 1) / C <= j) ++r;
                while (F * r / C > j) --r;
                imh[j] = *cl.map_shared_rank(&imh[j], r);
            }
        cl.sync();  // rank 0 has read the others' spectra
        if (rank != 0) return;
    }
    __syncthreads();
    if (imh_out)
        for (int j = tid; j < F; j += kThreads64) imh_out[(size_t)p * F + j] = imh[j];
    double term = 0.0;
    if (tid < G && (gates_out || ll_out)) {
        double acc = 0.0;
        for (int j = 0; j < F; ++j) acc += g_T[(size_t)tid * F + j] * imh[j];
        if (gates_out) gates_out[(size_t)p * G + tid] = acc;
        if (ll_out) {
            const double ea = eps_an[tid];
            const double v = ea * ea + (eps_mn * acc) * (eps_mn * acc);
            // models [s*obs_per, (s+1)*obs_per) share sounding s's data
            const double *yo = y_obs + (obs_per > 0 ? (size_t)(p / obs_per) * G : 0);
            const double rr = yo[tid] - acc;
            term = rr * rr / v + log(2.0 * kPi * v);
        }
    }
    if (ll_out) {
        if (warp * 32 < G) {
            const double t = warp_sum<double>(term);
            if (lane == 0) ll_part[warp] = t;
        }
        __syncthreads();
        if (tid == 0) {
            double acc = 0.0;
            for (int w = 0; w * 32 < G; ++w) acc += ll_part[w];
            ll_out[p] = -0.5 * acc;
        }
    }
}

int launch_forward_f64(const aem_system *sys, const aem_models_f64 *models, double *gates, double *imh,
                       const double *y_obs, int obs_per, const double *eps_an, double eps_mn, double *ll, void *stream,
                       const char *name, const int *active = nullptr, const int8_t *valid = nullptr) {
    if (!sys || !models) return fail(AEM_ERR_INVALID_ARG, std::string(name) + ": NULL system or models");
    if (models->n_models < 0 || models->lmax < 1 || models->lmax > AEM_MAX_LAYERS)
        return fail(AEM_ERR_INVALID_ARG, std::string(name) + ": n_models < 0 or lmax outside 1..AEM_MAX_LAYERS");
    if (models->n_models == 0) return AEM_OK;
    if (!gates && !imh && !ll) return fail(AEM_ERR_INVALID_ARG, std::string(name) + ": no output requested");
    if (!models->nlayers || !models->logsig || !models->logh || !models->m || !models->logtau || !models->c)
        return fail(AEM_ERR_INVALID_ARG, std::string(name) + ": NULL model array");
    if (ll && (!y_obs || !eps_an)) return fail(AEM_ERR_INVALID_ARG, std::string(name) + ": NULL y_obs or eps_an");
    const SystemTables &h = sys->host;
    const ModelsView<double> mv{models->n_models, models->lmax, models->nlayers, models->logsig, models->logh,
                                models->m, models->logtau, models->c};
    const size_t smem = smem_bytes_f64(h.F, h.K, models->lmax);
    // the largest any system needs, so that no caller lowers it under another
    AEM_CUDA_TRY(cudaFuncSetAttribute(forward_f64_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)smem_bytes_f64(AEM_MAX_FREQ, AEM_MAX_HANKEL, AEM_MAX_LAYERS)));
    // Models are split over clusters of up to eight CTAs until there are 16 CTAs
    // per SM to balance the last wave with (every CTA keeps at least two
    // frequencies).
    int C = 1;
    while (C < 8 && (long long)models->n_models * C < 16LL * sys->num_sms && h.F >= 4 * C) C *= 2;
    if ((long long)models->n_models * C > 0x7fffffffLL)
        return fail(AEM_ERR_INVALID_ARG, std::string(name) + ": too many models");
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(models->n_models * C), 1, 1);
    cfg.blockDim = dim3(kThreads64, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = (cudaStream_t)stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)C;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = C > 1 ? 1 : 0;
    AEM_CUDA_TRY(cudaLaunchKernelEx(&cfg, forward_f64_kernel, mv, h.F, h.G, h.K, h.cc_form,
                                    (const double *)sys->d_omega_d, (const double *)sys->d_lam_d,
                                    (const double *)sys->d_hw_d, (const double *)sys->d_T_d, (const double *)sys->d_tab64, gates,
                                    imh, y_obs, obs_per,
                                    eps_an, eps_mn, ll, active, valid));
    return AEM_OK;
}

// ===================================================================== FP32
// FP32 hot path.  Each thread carries TWO Hankel abscissae of the same
// frequency (k and k + K/2) through the layer recursion together, packed in
// 64-bit register pairs and advanced with the sm_100+ paired FP32 instructions
// (add/sub/mul/fma .f32x2): one issue slot per operation on both abscissae.
// The special functions (sqrt, rsqrt, rcp, ex2, sin, cos) stay scalar.
//
// The recursion is carried in w = sqrt(2) u.  Principal root of
// 2 (lambda^2 + s) with x = lambda^2 + Re s, y = Im s > 0 and m = |x + i y|:
//   t = m + |x|, rr = rsqrt(t); (t rr, y rr) is (Re w, Im w) when x >= 0 and
//   (Im w, Re w) otherwise.
// The interface coefficient comes from the two roots and their moduli alone,
//   r = (u_a - u_b) / (u_a + u_b) = (u_a - u_b) conj(u_a + u_b) / |u_a + u_b|^2
//     = [(m_a - m_b) + i (Im w_a Re w_b - Re w_a Im w_b)]
//       / [m_a + m_b + Re w_a Re w_b + Im w_a Im w_b]
// (|w|^2 = 2 m), nine paired operations and one reciprocal per abscissa where
// B / (w_a + w_b)^2 with B = 2 (s_a - s_b) takes fourteen and two more
// shared-memory records per interface.  Only Im R_0 is wanted; the rounding of
// m_a - m_b enters it multiplied by Im E of the layers above and is attenuated
// with the layer's own signal, and Im r keeps its relative accuracy, so the
// spectrum's error is lower than with the differenced s (FP32 emulation on 150
// random and 100 alternating stacks, relative to sum |w_k| |R_0|: largest
// 6.3e-7 against 1.4e-6, rms 4.0e-8 against 7.5e-8); the log-likelihood's by
// itself is not (see forward_f32_kernel's sums).
//   E = exp(-2 u h) = exp2(e w.x) (cos(e ln2 w.y) + i sin(e ln2 w.y)),
//   e = -sqrt(2) h log2(e).
// The Moebius step (N, D) <- (r D + N E, D + r N E) keeps R_0 = N / D.
// Lengths are counted in a power of two of the order of the system's 2 h + a
// (aem_system::len: lambda, s and h scaled by it exactly), so that |lambda^2 + s|^2
// and the product of two reciprocals' arguments stay inside the FP32 range
// whatever the geometry, for conductivities past any metal's.
using namespace f32x2;  // paired FP32 helpers and the hardware approximations (f32x2.h)

constexpr double kLn2Pi = 1.83787706640934548356;  // ln(2 pi)
constexpr int kDotParts = 4;  // warps that share a model's gate transform (every launch shape has them)

// The low part of a float pair; none beside an infinity or a NaN.
__device__ __forceinline__ float rest(float hi, float lo) { return fabsf(hi) <= 3.402823466e38f ? lo : 0.f; }

// rcoef2 for the air above the top layer: w_air = sqrt(2) lambda is real,
// m_air = lambda^2; nwair = -w_air.
__device__ __forceinline__ C2x2 rcoef2_air(u64 lam2, u64 nwair, const Root &b) {
    const u64 den = sub2(add2(lam2, b.m), mul2(nwair, b.re));
    const u64 ir = rcp2(den);
    C2x2 r;
    r.re = mul2(sub2(lam2, b.m), ir);
    r.im = mul2(mul2(nwair, b.im), ir);
    return r;
}

// he = ((e, e), (e ln2, e ln2)) of the layer below the interface.
// E = exp(-2 u h) of both abscissae as (Re, Im) pairs.
__device__ __forceinline__ void expm2(const Root &wb, ulonglong2 he, u64 &Ex, u64 &Ey) {
    float a0, a1;
    up2(mul2(he.x, wb.re), a0, a1);
    const u64 e = pk2(ex2_approx(a0), ex2_approx(a1));
#if AEM_F32_POLY_SINCOS
    u64 sn, cs;
    sincos2_poly(mul2(he.y, wb.im), sn, cs);
    Ex = mul2(e, cs);
    Ey = mul2(e, sn);
#else
    float f0, f1;
    up2(reduce_2pi2(mul2(he.y, wb.im)), f0, f1);
    float s0, c0, s1, c1;
    sincos_approx(f0, &s0, &c0);
    sincos_approx(f1, &s1, &c1);
    Ex = mul2(e, pk2(c0, c1));
    Ey = mul2(e, pk2(s0, s1));
#endif
}

__device__ __forceinline__ void mobius2(C2x2 &N, C2x2 &D, C2x2 r, const Root &wb, ulonglong2 he) {
    u64 Ex, Ey;
    expm2(wb, he, Ex, Ey);
    const u64 Px = sub2(mul2(N.re, Ex), mul2(N.im, Ey));
    const u64 Py = fma2(N.re, Ey, mul2(N.im, Ex));
    const u64 Nx = sub2(fma2(r.re, D.re, Px), mul2(r.im, D.im));
    const u64 Ny = fma2(r.re, D.im, fma2(r.im, D.re, Py));
    const u64 Dx = sub2(fma2(r.re, Px, D.re), mul2(r.im, Py));
    const u64 Dy = fma2(r.re, Py, fma2(r.im, Px, D.im));
    N.re = Nx;
    N.im = Ny;
    D.re = Dx;
    D.im = Dy;
}

// The first Moebius step, where D = 1: (N, D) <- (r + N E, 1 + r N E).
__device__ __forceinline__ void mobius2_d1(C2x2 &N, C2x2 &D, C2x2 r, const Root &wb, ulonglong2 he) {
    u64 Ex, Ey;
    expm2(wb, he, Ex, Ey);
    const u64 Px = sub2(mul2(N.re, Ex), mul2(N.im, Ey));
    const u64 Py = fma2(N.re, Ey, mul2(N.im, Ex));
    N.re = add2(r.re, Px);
    N.im = add2(r.im, Py);
    D.re = sub2(fma2(r.re, Px, kOne2), mul2(r.im, Py));
    D.im = fma2(r.re, Py, mul2(r.im, Px));
}

// A load of the records or exponents by shared-memory address.  It is volatile
// but clobbers no memory: what orders it after the stores is the barrier between
// them and the empty clobber that opens every item (item_of).
__device__ __forceinline__ ulonglong2 lds16(unsigned a) {
    ulonglong2 v;
    asm volatile("ld.shared.v2.u64 {%0, %1}, [%2];" : "=l"(v.x), "=l"(v.y) : "r"(a));
    return v;
}

// Im R_0 for the two abscissae of one work item.  rec, he: shared-memory
// addresses of the frequency's layer records and of the layers' exponents.
// LT > 0: the layer count is the compile-time LT and the layer loop is
// unrolled completely; LT = 0: the runtime L, two layers per iteration.
template <int LT>
__device__ __forceinline__ void im_r0_pair(u64 lam2, u64 nwair, unsigned rec, unsigned he, int L_rt, float &out0,
                                           float &out1) {
    const int L = LT > 0 ? LT : L_rt;
    unsigned rp = rec + 16u * (unsigned)(L - 1);
    Root wb = root2(lam2, lds16(rp));
    if (L == 1) {
        up2(rcoef2_air(lam2, nwair, wb).im, out0, out1);
        return;
    }
    rp -= 16;
    Root wa = root2(lam2, lds16(rp));
    C2x2 N = rcoef2(wa, wb), D;
    if (L == 2) {
        mobius2_d1(N, D, rcoef2_air(lam2, nwair, wa), wa, lds16(he));
    } else if constexpr (LT > 2) {
#pragma unroll
        for (int n = LT - 3; n >= 0; --n) {
            wb = root2(lam2, lds16(rec + 16 * n));
            if (n == LT - 3)
                mobius2_d1(N, D, rcoef2(wb, wa), wa, lds16(he + 16 * (n + 1)));
            else
                mobius2(N, D, rcoef2(wb, wa), wa, lds16(he + 16 * (n + 1)));
            wa = wb;
            // each step's shared-memory loads stay in their step (hoisting
            // them ahead raises the register pressure into spills)
            asm volatile("" ::: "memory");
        }
        mobius2(N, D, rcoef2_air(lam2, nwair, wa), wa, lds16(he));
    } else {
        unsigned hp = he + 16u * (unsigned)(L - 2);
        rp -= 16;
        wb = root2(lam2, lds16(rp));
        mobius2_d1(N, D, rcoef2(wb, wa), wa, lds16(hp));
        // wb is layer L - 3; the layers above it come in pairs, so that the
        // roots swap roles without a copy
        if (L & 1) {
            wa = wb;
        } else {
            rp -= 16;
            hp -= 16;
            wa = root2(lam2, lds16(rp));
            mobius2(N, D, rcoef2(wa, wb), wb, lds16(hp));
        }
#pragma unroll 1
        while (rp != rec) {
            wb = root2(lam2, lds16(rp - 16));
            mobius2(N, D, rcoef2(wb, wa), wa, lds16(hp - 16));
            wa = root2(lam2, lds16(rp - 32));
            mobius2(N, D, rcoef2(wa, wb), wb, lds16(hp - 32));
            rp -= 32;
            hp -= 32;
        }
        mobius2(N, D, rcoef2_air(lam2, nwair, wa), wa, lds16(he));
    }
    float n0, n1, d0, d1;
    up2(sub2(mul2(N.im, D.re), mul2(N.re, D.im)), n0, n1);
    up2(fma2(D.re, D.re, mul2(D.im, D.im)), d0, d1);
    out0 = n0 * rcp_approx(d0);
    out1 = n1 * rcp_approx(d1);
}

// Claiming the next model from the grid itself (cluster launch control): with
// one CTA per model in the grid, a running CTA cancels the next one that has
// not been started yet and takes over its index, so CTAs stay resident and
// whichever is free takes the next model, with no counter in memory to
// allocate, reset or keep apart between streams (a launch without a recorded
// shape allocates nothing).  One thread asks (asynchronously, answered into
// shared memory) and later reads the answer.  A counter is about 1 % faster
// (9.19 against 9.27 ms for 2^17 models of the 60 x 200 system), so the
// recorded dynamic shapes and the callers that own one keep it.
struct alignas(16) Claim {
    unsigned long long answer[2];
    unsigned long long bar;
    unsigned parity;
};
constexpr unsigned kClaimSpins = 1u << 22;  // a bound on the wait; an answer takes about a microsecond

__device__ __forceinline__ void claim_init(Claim *c) {
    c->parity = 0;
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"((unsigned)__cvta_generic_to_shared(&c->bar)) : "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
__device__ __forceinline__ void claim_ask(Claim *c) {
    const unsigned a = (unsigned)__cvta_generic_to_shared(c->answer), b = (unsigned)__cvta_generic_to_shared(&c->bar);
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // the last answer has been read
    asm volatile("{\n\t.reg .b64 t;\n\tmbarrier.arrive.expect_tx.shared::cta.b64 t, [%0], 16;\n\t}" ::"r"(b) : "memory");
    asm volatile(
        "clusterlaunchcontrol.try_cancel.async.shared::cta.mbarrier::complete_tx::bytes.b128 [%0], [%1];" ::"r"(a),
        "r"(b)
        : "memory");
}
// At most limit - 1 polls of the answer's barrier.
__device__ __forceinline__ bool claim_wait(unsigned bar, unsigned parity, unsigned limit) {
    unsigned ok = 0;
    for (unsigned i = 1; i < limit && !ok; ++i)
        asm volatile(
            "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(ok)
            : "r"(bar), "r"(parity)
            : "memory");
    return ok != 0;
}
// The index taken over, or n when none is left.  A wait that runs out is
// recorded in *status and waited for once more: the request is in flight
// into this CTA's shared memory, and the CTA it cancels has left its model to
// this one.  Should that wait run out too, the launch ends without the models
// of this CTA's answer (and the context should be treated as unreliable).
__device__ __forceinline__ int claim_answer(Claim *c, int n, int *status, unsigned limit) {
    const unsigned a = (unsigned)__cvta_generic_to_shared(c->answer), b = (unsigned)__cvta_generic_to_shared(&c->bar);
    const unsigned parity = c->parity;
    c->parity = parity ^ 1;
    if (!claim_wait(b, parity, limit)) {
        atomicExch(status, (int)AEM_ERR_TIMEOUT);
        if (!claim_wait(b, parity, kClaimSpins)) return n;
    }
    unsigned got, x;
    asm volatile(
        "{\n\t.reg .b128 r;\n\t.reg .pred p;\n\t.reg .b32 y, z, w;\n\tld.shared.b128 r, [%2];\n\t"
        "clusterlaunchcontrol.query_cancel.is_canceled.pred.b128 p, r;\n\tselp.u32 %0, 1, 0, p;\n\tmov.u32 %1, 0;\n\t"
        "@p clusterlaunchcontrol.query_cancel.get_first_ctaid.v4.b32.b128 {%1, y, z, w}, r;\n\t}"
        : "=r"(got), "=&r"(x)
        : "r"(a)
        : "memory");
    return got ? (int)x : n;
}

// The per-item value buffer: kValsWords floats (24 KB), the same for every
// launch shape, so that the Hankel sums come out identical whatever the
// shape, the scheduling or the row stride (lmax) of the models.
constexpr int kValsWords = 6144;
static_assert(kValsWords % 32 == 0, "rounds must end on a whole group");

// Words of the buffer one system uses: all of it, or its single round's items.
__host__ __device__ inline int vals_words(int F, int K2) {
    const int n = (F * K2 + 31) & ~31;
    return n < kValsWords ? n : kValsWords;
}

// Shared memory (dynamic), in order: REC[F*LS] (ulonglong2: per frequency and
// layer the (Re s, Re s) and (Im s, Im s) pairs), KR[K2] (ulonglong2: per
// abscissa pair the (lambda^2, -sqrt(2) lambda) pairs), HW[K2] (the pairs'
// Hankel weights), vals[vals_words], imh[F] (float pairs), Ts[F*G] (T by
// frequency), bound[G] (d_T_pair's), TH[F*LS] (float: the depth cutoff's
// thresholds).  The items (frequency major, F*K2 of
// them) are taken in rounds of kValsWords: every item stores its weighted pair
// value at its own index in the buffer; after the round each frequency the
// round touched is summed by four consecutive lanes (lane s adds the values at
// s + 4 i into four accumulators by i mod 4, then a tree over the sixteen
// partial sums, two levels by shuffles) and added to imh[f], rounds in order.
// From the sixteen partial sums on the sums are float pairs (TwoSum), and so
// is the transform: the gates cancel to about a hundredth of their terms, and
// with the spectrum and T rounded to a float and a plain dot product these
// three made most of the log-likelihood's error.  On 256 models about one
// earth (40 frequencies, 120 abscissae, up to 8 layers) it is 5.4e-7 of the
// norm against 64 bits, 1.1e-6 without (1.3e-6 with the differenced s before
// that); on the 60 x 200 system 4.4e-7 against 1.3e-6, and the gradient's
// error falls with it by 2 to 4.  32,768 models of the former: 0.94 ms, 0.91
// without (0.95 with TwoProd and TwoSum).
// The order of every sum is fixed by the item indices alone.  (The throughput
// system's 60 x 100 items take one round.)
// DYN: models in a fixed order (0), claimed from work_counter (1) or from the
// grid, which then has a CTA per model (2).
template <int NT, int MINB, int DYN, bool SPEC>
__global__ void __launch_bounds__(NT, MINB) forward_f32_kernel(ModelsView<float> mv, int F, int G, int K,
                                                               int cc_form, int LS, float len,
                                                               const float *__restrict__ g_omega,
                                                               const float2 *__restrict__ g_wmu,
                                                               const float *__restrict__ g_lam,
                                                               const float *__restrict__ g_hw,
                                                               const float2 *__restrict__ g_T,
                                                               float *__restrict__ gates_out,
                                                               float *__restrict__ imh_out,
                                                               const double *__restrict__ y_obs, int obs_per,
                                                               const double *__restrict__ eps_an, double eps_mn,
                                                               double *__restrict__ ll_out,
                                                               int *__restrict__ work_counter,
                                                               int *__restrict__ status, unsigned claim_limit,
                                                               const int *__restrict__ active, float att0,
                                                               unsigned long long *__restrict__ steps_out,
                                                               const int8_t *__restrict__ valid) {
    if (active && *active == 0) return;  // a gated launch the caller switched off on the device
    constexpr int NW = NT / 32;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int K2 = (K + 1) / 2;
    ulonglong2 *REC = reinterpret_cast<ulonglong2 *>(smem_raw);
    ulonglong2 *KR = REC + (size_t)F * LS;
    u64 *HW = reinterpret_cast<u64 *>(KR + K2);
    float *vals = reinterpret_cast<float *>(HW + K2);
    float2 *imh = reinterpret_cast<float2 *>(vals + vals_words(F, K2));
    float *Ts = reinterpret_cast<float *>(imh + F), *bound = Ts + (size_t)G * F;
    float *TH = bound + G;  // depth-cutoff thresholds, [F][LS]
    __shared__ ulonglong2 HE[AEM_MAX_LAYERS];
    __shared__ float lh[AEM_MAX_LAYERS];
    __shared__ float lsig[AEM_MAX_LAYERS], lm[AEM_MAX_LAYERS], ltau[AEM_MAX_LAYERS], lc[AEM_MAX_LAYERS];
    __shared__ float lsp[AEM_MAX_LAYERS], lcp[AEM_MAX_LAYERS];
    __shared__ double ll_part[2];
    __shared__ float2 gate_part[kDotParts][AEM_MAX_GATES];
    __shared__ unsigned imh_max;  // the largest |Im H| of the model, as its bits

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (int i = tid; i < G * (F + 1); i += blockDim.x) Ts[i] = g_T[i].x;
    // abscissa pairs (k, k + K2); an odd K pads the last pair with a zero weight
    for (int k = tid; k < K2; k += blockDim.x) {
        const int kb = k + K2 < K ? k + K2 : K - 1;
        const float la = g_lam[k], lb = g_lam[kb];
        KR[k] = make_ulonglong2(pk2(la * la, lb * lb),
                                pk2(-1.41421356237309505f * la, -1.41421356237309505f * lb));
        HW[k] = pk2(g_hw[k], k + K2 < K ? g_hw[kb] : 0.f);
    }
    const unsigned rec_a = (unsigned)__cvta_generic_to_shared(REC), he_a = (unsigned)__cvta_generic_to_shared(HE);
    const float ilen = 1.f / len;
    const int FK2 = F * K2;
    const bool wide = K2 >= 32;  // 32 consecutive items span two frequencies at most

    __shared__ int next_model;
    __shared__ Claim claim;
    if (DYN == 2 && tid == 0) claim_init(&claim);
    unsigned int nsteps = 0;  // layer-steps of the groups this lane bucketed (steps_out)
    for (int p = blockIdx.x; p < mv.n; p = DYN ? next_model : p + gridDim.x) {
        const int L = mv.nlayers[p];
        __syncthreads();
        // The next model is claimed when this one's items are done, not before:
        // what is left at the end then goes to whichever CTA is free, not to
        // those that started first (1,300 models on 1,216 resident CTAs: 75 us
        // claimed at the model's start, 60 us).
        auto ask = [&] {
            if (DYN == 1 && tid == 0) next_model = (int)gridDim.x + atomicAdd(work_counter, 1);
            if (DYN == 2 && tid == 0) claim_ask(&claim);
        };
        auto claimed = [&] {  // into next_model, before a barrier
            if (DYN == 2 && tid == 0) next_model = claim_answer(&claim, mv.n, status, claim_limit);
        };
        if (valid && !valid[p]) {  // a proposal the caller will not use (CTA-uniform)
            ask();
            claimed();
            if (DYN) __syncthreads();  // next_model visible to every thread
            continue;
        }
        if (tid < L) {
            const size_t o = (size_t)p * mv.lmax + tid;
            lsig[tid] = exp10f(mv.logsig[o]);
            lh[tid] = exp10f(mv.logh[o]) * ilen;
            const float e = -1.41421356237309505f * 1.44269504088896341f * lh[tid];
            HE[tid] = make_ulonglong2(pk2(e, e), pk2(e * 0.69314718055994531f, e * 0.69314718055994531f));
            lm[tid] = mv.m[o];
            ltau[tid] = exp10f(mv.logtau[o]);
            lc[tid] = mv.c[o];
            float sp, cp;
            sincospif(0.5f * mv.c[o], &sp, &cp);
            lsp[tid] = sp;
            lcp[tid] = cp;
        }
        for (int j = tid; j < F; j += blockDim.x) imh[j] = make_float2(0.f, 0.f);
        if (tid == 0) imh_max = 0u;
        __syncthreads();
        // Cole-Cole per (frequency, layer): x = (w tau)^c e^{i pi c / 2}, s = i w mu0 sigma
        for (int i = tid; i < F * L; i += blockDim.x) {
            const int f = i / L, n = i - f * L;
            const float w = g_omega[f];
            const float sig = lsig[n], mm = lm[n];
            float sr = sig, si = 0.f;
            if (mm != 0.f) {
                const float cc = lc[n];
                const float mag = expf(cc * logf(w * ltau[n]));
                const float sp = lsp[n], cp = lcp[n];
                const float xr = 1.f + mag * cp, xi = mag * sp;
                const float den = xr * xr + xi * xi;
                // Each form is evaluated without cancellation.  The paper's
                // sigma_inf (1 - m / (1 + x)) as 1 - m Re(1/(1+x)) loses the
                // digits of 1 - m when m -> 1 at small w tau (a relative error
                // of 2^-24 / (1 - m) in Re sigma, up to 3e-5 of the Hankel
                // sum on the random-model workload); written as
                // ((1 - m) + x) / (1 + x), with 1 - m exact for m >= 1/2, every
                // real part is a sum of non-negative terms (c <= 1 so Re x >= 0)
                // and every imaginary part is a single product m Im x / |.|^2.
                if (cc_form == AEM_CC_PAPER) {
                    sr = sig * (fmaf((1.f - mm) + mag * cp, xr, xi * xi) / den);
                    si = sig * (mm * xi / den);
                } else if (cc_form == AEM_CC_LITERAL) {
                    const float br = 1.f + (1.f - mm) * mag * cp, bi = (1.f - mm) * mag * sp;
                    sr = sig * (fmaf(br, xr, bi * xi) / den);
                    si = -sig * (mm * xi / den);
                } else {
                    const float br = 1.f + (1.f - mm) * mag * cp, bi = (1.f - mm) * mag * sp;
                    const float bd = br * br + bi * bi;
                    sr = sig * (fmaf(xr, br, xi * bi) / bd);
                    si = sig * (mm * xi / bd);
                }
            }
            // w mu0 as a float pair: one rounding is left, that of the product
            const float2 wm = g_wmu[f];
            const float sx = -fmaf(wm.x, si, wm.y * si), sy = fmaf(wm.x, sr, wm.y * sr);
            REC[(size_t)f * LS + n] = make_ulonglong2(pk2(sx, sx), pk2(sy, sy));
        }
        __syncthreads();
        // the depth cutoff's thresholds (depth_cutoff.h), one frequency per thread
        const bool cut = att0 > 0.f && L > 1;
        if (cut)
            for (int f = tid; f < F; f += blockDim.x) {
                const float4 *rf = reinterpret_cast<const float4 *>(REC + (size_t)f * LS);
                depth_thresholds([&](int n) { const float4 v = rf[n]; return make_float2(v.x, v.z); }, lh, L, att0,
                                 TH + (size_t)f * LS);
            }
        __syncthreads();

        // The item loop in rounds of kValsWords items.  A warp takes whole
        // groups of 32 consecutive items (one per lane), the same groups in
        // every launch shape: its groups of the round are g = g0 + warp + j NW,
        // looked at 32 at a time, one per lane.  Each lane finds its group's
        // layer count: the largest any of its items needs, which within a
        // frequency is that of its smallest lambda (the pair's first abscissa),
        // so the group's first item and the first item of each later frequency
        // it reaches.
        for (int r0 = 0; r0 < FK2; r0 += kValsWords) {
            const int r1 = r0 + kValsWords < FK2 ? r0 + kValsWords : FK2;
            const int g0 = r0 >> 5, g1 = (r1 + 31) >> 5;
            for (int gc = g0 + warp; gc < g1; gc += 32 * NW) {
                const int gl = gc + lane * NW;
                int lpl = 0, pkl = 0;
                if (gl < g1) {
                    const int first = 32 * gl, last = min(first + 31, FK2 - 1);
                    const int f0 = first / K2, f1 = last / K2;
                    pkl = (f0 << 16) | (first - f0 * K2);
                    lpl = L;
                    if (cut) {
                        lpl = 1;
                        for (int ff = f0; ff <= f1; ++ff) {
                            float l2, lb2;
                            up2(KR[ff == f0 ? first - f0 * K2 : 0].x, l2, lb2);
                            lpl = max(lpl, depth_layers(l2, TH + (size_t)ff * LS, L));
                        }
                    }
                    if (steps_out) nsteps += (unsigned int)lpl * (unsigned int)(last + 1 - first);
                }
                auto item_of = [&](int pk, int j, auto body) {
                    const int item = 32 * (gc + j * NW) + lane;
                    if (item >= r1) return;
                    int f = (pk >> 16) & 0xff, k = (pk & 0xffff) + lane;
                    if (k >= K2) {  // into the next frequency; further ones only when K2 < 32
                        k -= K2;
                        ++f;
                        if (!wide)
                            while (k >= K2) {
                                k -= K2;
                                ++f;
                            }
                    }
                    const ulonglong2 lw = KR[k];
                    float v0, v1;
                    asm volatile("" ::: "memory");  // lds16
                    body(lw, rec_a + (unsigned)(f * LS) * 16u, v0, v1);
                    float h0, h1;
                    up2(HW[k], h0, h1);
                    vals[item - r0] = fmaf(h0, v0, h1 * v1);
                };
                if constexpr (SPEC) {
                    // bucket by bucket of layer count (a ballot per count), so
                    // every bucket runs the recursion unrolled for its count
                    for (int v = __reduce_max_sync(kFull, lpl); v >= 1; --v) {
                        const unsigned int all = __ballot_sync(kFull, lpl == v);
                        if (!all) continue;
                        auto run = [&](auto lt) {
                            constexpr int LT = decltype(lt)::value;
                            for (unsigned int mask = all; mask; mask &= mask - 1) {
                                const int jl = __ffs(mask) - 1;
                                const int pk = __shfl_sync(kFull, pkl, jl);
                                item_of(pk, jl, [&](ulonglong2 lw, unsigned rec, float &v0, float &v1) {
                                    im_r0_pair<LT>(lw.x, lw.y, rec, he_a, v, v0, v1);
                                });
                            }
                        };
                        switch (v) {
                            case 1: run(std::integral_constant<int, 1>{}); break;
                            case 2: run(std::integral_constant<int, 2>{}); break;
                            case 3: run(std::integral_constant<int, 3>{}); break;
                            case 4: run(std::integral_constant<int, 4>{}); break;
                            case 5: run(std::integral_constant<int, 5>{}); break;
                            case 6: run(std::integral_constant<int, 6>{}); break;
                            case 7: run(std::integral_constant<int, 7>{}); break;
                            case 8: run(std::integral_constant<int, 8>{}); break;
                            case 9: run(std::integral_constant<int, 9>{}); break;
                            case 10: run(std::integral_constant<int, 10>{}); break;
                            default: run(std::integral_constant<int, 0>{}); break;
                        }
                    }
                } else {
                    pkl |= lpl << 24;
                    const int nj = min(32, (g1 - gc + NW - 1) / NW);
                    for (int j = 0; j < nj; ++j) {
                        const int pk = __shfl_sync(kFull, pkl, j);
                        item_of(pk, j, [&](ulonglong2 lw, unsigned rec, float &v0, float &v1) {
                            im_r0_pair<0>(lw.x, lw.y, rec, he_a, pk >> 24, v0, v1);
                        });
                    }
                }
            }
            if (r1 == FK2) ask();
            __syncthreads();
            // the round's share of each frequency's Hankel sum, in a fixed
            // order: four consecutive lanes per frequency; lane s adds the
            // values at a + s + 4 i into four accumulators by i mod 4 (the
            // sixteen interleaved subsets of the frequency's values, each of
            // them spread over its whole abscissa range, so partial sums
            // cancel as the whole does), then (c0 + c1) + (c2 + c3) and two
            // shuffles (one round, the throughput systems' case: frequencies
            // 0..F-1)
            const int fa = r0 == 0 ? 0 : r0 / K2, fb = r1 == FK2 ? F - 1 : (r1 - 1) / K2;
            for (int t0 = 0; t0 < 4 * (fb - fa + 1); t0 += blockDim.x) {  // CTA-uniform trip count
                const int t = t0 + tid, j = fa + (t >> 2), s = t & 3;
                float acc = 0.f, err = 0.f;
                if (j <= fb) {
                    const int a = j * K2 > r0 ? j * K2 : r0, b = (j + 1) * K2 < r1 ? (j + 1) * K2 : r1;
                    const float *vq = vals - r0;
                    float c0 = 0.f, c1 = 0.f, c2 = 0.f, c3 = 0.f;
                    for (int q = a + s; q < b; q += 16) {
                        c0 += vq[q];
                        if (q + 4 < b) c1 += vq[q + 4];
                        if (q + 8 < b) c2 += vq[q + 8];
                        if (q + 12 < b) c3 += vq[q + 12];
                    }
                    float e0, e1;
                    two_sum(c0, c1, c0, e0);
                    two_sum(c2, c3, c2, e1);
                    two_sum(c0, c2, acc, err);
                    err += e0 + e1;
                }
#pragma unroll
                for (int o = 1; o <= 2; o <<= 1) {
                    float e;
                    two_sum(acc, __shfl_xor_sync(kFull, acc, o), acc, e);
                    err += __shfl_xor_sync(kFull, err, o);
                    err += e;
                }
                unsigned bits = 0u;
                if (s == 0 && j <= fb) {
                    const float2 had = imh[j];
                    float h, e;
                    two_sum(had.x, acc, h, e);
                    imh[j] = make_float2(h, rest(h, had.y + (err + e)));
                    bits = __float_as_uint(fabsf(h));
                }
                bits = __reduce_max_sync(kFull, bits);
                if (lane == 0) atomicMax(&imh_max, bits);
            }
            if (r1 == FK2) claimed();
            __syncthreads();
        }

        // gates: dot products in float pairs, a quarter of the frequencies per
        // warp, lane = gate.  The sum begins at a power of two above all its
        // partial sums, so that what it rounds off of a product is exact (Dekker's
        // Fast2Sum): t x - (sum after - sum before), six operations a term
        // where TwoProd and TwoSum take thirteen.  T's low parts are read from
        // global memory: beside the high ones they would cost systems of many
        // gates and frequencies a resident CTA (64 x 128 x 200, 8,000 models:
        // 2.32 ms against 1.62).
        if (warp < kDotParts && (gates_out || ll_out)) {
            const int j0 = F * warp / kDotParts, j1 = F * (warp + 1) / kDotParts;
            const float xmax = __uint_as_float(imh_max);
            for (int g = lane; g < G; g += 32) {
                const float top = bound[g] * xmax;  // >= sum_j |t_j x_j|
                const float base = __uint_as_float(min((__float_as_uint(top) >> 23) + 2u, 254u) << 23);
                float acc = base, err = 0.f;
#pragma unroll 4
                for (int j = j0; j < j1; ++j) {
                    const float t = Ts[j * G + g], lo = __ldg(&g_T[j * G + g].y);
                    const float2 x = imh[j];
                    const float sum = fmaf(t, x.x, acc);
                    err = fmaf(t, x.y, fmaf(lo, x.x, err)) + fmaf(t, x.x, acc - sum);
                    acc = sum;
                }
                gate_part[warp][g] = make_float2(acc - base, err);
            }
        }
        if (gates_out || ll_out) __syncthreads();
        double term = 0.0;
        if (tid < G && (gates_out || ll_out)) {
            float acc = 0.f, err = 0.f;
#pragma unroll
            for (int w = 0; w < kDotParts; ++w) {
                const float2 v = gate_part[w][tid];
                float e;
                two_sum(acc, v.x, acc, e);
                err += v.y + e;
            }
            err = rest(acc, err);
            const float gate = acc + err;
            if (gates_out) gates_out[(size_t)p * G + tid] = gate;
            if (ll_out) {
                const double *yo = y_obs + (obs_per > 0 ? (size_t)(p / obs_per) * G : 0);
                // FP32 terms (the residual from an FP64 difference, the
                // variance, one division and one logarithm), FP64 sum: FP64
                // terms cost this serial epilogue 1 % of the whole launch
                const float r = (float)(yo[tid] - (double)acc) - err;
                const float ea = (float)eps_an[tid], q = (float)eps_mn * gate;
                const float v = fmaf(q, q, ea * ea);
                term = (double)(__fdiv_rn(r * r, v) + logf(v)) + kLn2Pi;
            }
        }
        if (imh_out)
            for (int j = tid; j < F; j += blockDim.x) imh_out[(size_t)p * F + j] = imh[j].x + imh[j].y;
        if (ll_out) {
            if (G <= 32) {
                // every term is in warp 0: its tree is the whole sum (0 + t = t
                // exactly, as the general form below would add it), no barrier
                if (warp == 0) {
                    const double t = warp_sum<double>(term);
                    if (lane == 0) ll_out[p] = -0.5 * t;
                }
            } else {
                if (warp * 32 < G) {
                    const double t = warp_sum<double>(term);
                    if (lane == 0) ll_part[warp] = t;
                }
                __syncthreads();
                if (tid == 0) {
                    double acc = 0.0;
                    for (int w = 0; w * 32 < G; ++w) acc += ll_part[w];
                    ll_out[p] = -0.5 * acc;
                }
            }
        }
    }
    if (steps_out) {
        const unsigned long long t = warp_sum<unsigned long long>(nsteps);
        if (lane == 0) atomicAdd(steps_out, t);
    }
}

size_t smem_bytes_f32(int F, int G, int K, int LS) {
    const int K2 = (K + 1) / 2;
    return sizeof(ulonglong2) * ((size_t)F * LS + K2) + sizeof(u64) * (size_t)K2 +
           sizeof(float) * (vals_words(F, K2) + 2 * (size_t)F + (size_t)G * (F + 1) + (size_t)F * LS);
}

// Launch shapes of forward_f32_kernel: threads per CTA, resident CTAs per SM
// the register budget must allow, and whether the recursion is unrolled per
// layer count.  A marginal layer costs a warp's 32 items about 96 cycles of an
// SM sub-partition unrolled and 104 in the two-layer loop (register-port and
// special-function rates together, whatever the shape), but the unrolled code
// (about 55 steps) overflows the instruction cache when many small CTAs are
// each at another layer count, while the small CTAs lose less at the barriers
// between a model's phases.  2^17 random models of the 60-frequency,
// 200-abscissa system, dynamic: 9.36 ms unrolled at 256 x 3, 10.8 ms looped at 128 x 8;
// 32,768 models of the 40-frequency, 120-abscissa one (up to 8 layers): 1.03
// and 0.92 ms.  (10.34 and 1.07 ms before the interface coefficient of the
// roots alone, all unrolled.)
struct F32Shape {
    int nt, minb;
};
#define AEM_SHAPES(X)                                                                        \
    X(0, 256, 4, false) X(1, 128, 8, false) X(2, 512, 2, true) X(3, 256, 3, true) X(4, 128, 6, false)
#define AEM_SHAPE(I, NT, MINB, SPEC) {NT, MINB},
constexpr F32Shape kF32Shapes[] = {AEM_SHAPES(AEM_SHAPE)};
#undef AEM_SHAPE
// shapes kNumBase .. 2 kNumBase - 1 are the same with dynamic model scheduling
constexpr int kNumBase = sizeof(kF32Shapes) / sizeof(kF32Shapes[0]);
constexpr int kNumF32Shapes = 2 * kNumBase;
// shapes 0 and 1 taking their models from the grid, for launches without a recorded shape
constexpr int kFromGrid = kNumF32Shapes;
static_assert(kNumF32Shapes == AEM_F32_SHAPES, "");

template <int IDX, int NT, int MINB, int DYN, bool SPEC>
int launch_shape(const aem_system *sys, const ModelsView<float> &mv, int LS, float *gates, float *imh,
                 const double *y_obs, int obs_per, const double *eps_an, double eps_mn, double *ll,
                 cudaStream_t stream, int *counter_ext, const int *active, unsigned long long *steps,
                 const int8_t *valid) {
    const SystemTables &h = sys->host;
    auto kern = forward_f32_kernel<NT, MINB, DYN, SPEC>;
    const size_t smem = smem_bytes_f32(h.F, h.G, h.K, LS);
    int per_sm = 0;
    if (const int rc = resident_ctas(&sys->fwd_ctas[IDX][LS], kern, NT, smem, sys->device, &per_sm)) return rc;
    if (per_sm < 1) return fail(AEM_ERR_UNSUPPORTED, "forward kernel: launch shape does not fit on an SM");
    long long grid = (long long)sys->num_sms * per_sm;
    if (grid > mv.n || DYN == 2) grid = mv.n;
    int *counter = counter_ext;
    const bool own = DYN == 1 && !counter_ext;
    if (own)  // stream-ordered: one counter per launch, so launches on other streams never share it
        AEM_CUDA_TRY(cudaMallocAsync((void **)&counter, sizeof(int), stream));
    if (DYN == 1) AEM_CUDA_TRY(cudaMemsetAsync(counter, 0, sizeof(int), stream));
    kern<<<(unsigned)grid, NT, smem, stream>>>(mv, h.F, h.G, h.K, h.cc_form, LS, sys->len, sys->d_omega_f,
                                               sys->d_wmu_f, sys->d_lamu_f, sys->d_hw_f, sys->d_T_pair, gates, imh, y_obs, obs_per, eps_an, eps_mn,
                                               ll, counter, sys->d_status,
                                               sys->wait_spins ? sys->wait_spins : kClaimSpins, active, sys->depth_att, steps, valid);
    const cudaError_t e = cudaGetLastError();
    if (own) cudaFreeAsync(counter, stream);
    AEM_CUDA_TRY(e);
    return AEM_OK;
}

int launch_shape_index(int idx, const aem_system *sys, const ModelsView<float> &mv, int LS, float *gates,
                       float *imh, const double *y_obs, int obs_per, const double *eps_an, double eps_mn, double *ll,
                       cudaStream_t stream, int *counter_ext = nullptr, const int *active = nullptr,
                       unsigned long long *steps = nullptr, const int8_t *valid = nullptr) {
#define AEM_SHAPE_CASE(I, NT, MINB, DYN, SPEC)                                                                     \
    case I:                                                                                                        \
        return launch_shape<I, NT, MINB, DYN, SPEC>(sys, mv, LS, gates, imh, y_obs, obs_per, eps_an, eps_mn, ll,   \
                                                    stream, counter_ext, active, steps, valid);
#define AEM_SHAPE(I, NT, MINB, SPEC)         \
    AEM_SHAPE_CASE(I, NT, MINB, 0, SPEC)     \
    AEM_SHAPE_CASE(I + kNumBase, NT, MINB, 1, SPEC)
    switch (idx) {
        AEM_SHAPES(AEM_SHAPE)
        AEM_SHAPE_CASE(kFromGrid, 256, 4, 2, false)
        AEM_SHAPE_CASE(kFromGrid + 1, 128, 8, 2, false)
        default: return fail(AEM_ERR_INVALID_ARG, "forward kernel: launch shape");
    }
#undef AEM_SHAPE
#undef AEM_SHAPE_CASE
}

// The launch shape of n_models models with row stride LS: the recorded one, or
// else the rule's.  counter: the caller has a work counter.
int shape_of_launch(const aem_system *sys, int LS, int n_models, bool counter, int *out) {
    // No shape recorded.  At most two models per SM: the largest CTAs, which
    // finish a model soonest.  Otherwise the looped shape of which more threads
    // are resident (the value buffer of many frequencies and abscissae leaves
    // room for fewer CTAs), the smaller one on a tie, with dynamic scheduling
    // once there are more models than resident CTAs.  3,001 and 20,000 models of
    // up to 10 layers of the 60 x 200 system: 341 and 1950 us at 128 x 8 in
    // fixed order, 260 and 1486 us; up to 8 layers of the 40 x 120 system, where
    // 128 x 8 stays: 120 and 654 us, 108 and 555 us.
    int shape = sys->f32_shape[LS];
    if (shape < 0) {
        if (n_models <= 2 * sys->num_sms) {
            shape = 2;
        } else {
            const size_t smem = smem_bytes_f32(sys->host.F, sys->host.G, sys->host.K, LS);
            int n0 = 0, n1 = 0;
            if (const int rc = resident_ctas(&sys->fwd_ctas[kFromGrid][LS], forward_f32_kernel<256, 4, 2, false>, 256,
                                             smem, sys->device, &n0))
                return rc;
            if (const int rc = resident_ctas(&sys->fwd_ctas[kFromGrid + 1][LS], forward_f32_kernel<128, 8, 2, false>,
                                             128, smem, sys->device, &n1))
                return rc;
            shape = n1 >= 2 * n0 ? 1 : 0;
            if (n_models > (long long)sys->num_sms * (shape ? n1 : n0))
                shape += counter ? kNumBase : kFromGrid;
        }
    }
    *out = shape;
    return AEM_OK;
}

template <class Models>
int launch_forward_f32(const aem_system *sys, const Models *models, float *gates, float *imh, const double *y_obs,
                       int obs_per, const double *eps_an, double eps_mn, double *ll, void *stream, const char *name,
                       int *counter_ext = nullptr, const int *active = nullptr,
                       unsigned long long *steps = nullptr, const int8_t *valid = nullptr) {
    if (!sys || !models) return fail(AEM_ERR_INVALID_ARG, std::string(name) + ": NULL system or models");
    if (models->n_models < 0 || models->lmax < 1 || models->lmax > AEM_MAX_LAYERS)
        return fail(AEM_ERR_INVALID_ARG, std::string(name) + ": n_models < 0 or lmax outside 1..AEM_MAX_LAYERS");
    if (models->n_models == 0) return AEM_OK;
    if (!gates && !imh && !ll) return fail(AEM_ERR_INVALID_ARG, std::string(name) + ": no output requested");
    if (!models->nlayers || !models->logsig || !models->logh || !models->m || !models->logtau || !models->c)
        return fail(AEM_ERR_INVALID_ARG, std::string(name) + ": NULL model array");
    if (ll && (!y_obs || !eps_an)) return fail(AEM_ERR_INVALID_ARG, std::string(name) + ": NULL y_obs or eps_an");
    ModelsView<float> mv{models->n_models, models->lmax, models->nlayers, models->logsig, models->logh,
                           models->m, models->logtau, models->c};
    const int LS = models->lmax;
    int shape = 0;
    if (const int rc = shape_of_launch(sys, LS, models->n_models, counter_ext != nullptr, &shape)) return rc;
    return launch_shape_index(shape, sys, mv, LS, gates, imh, y_obs, obs_per, eps_an, eps_mn, ll,
                              (cudaStream_t)stream, counter_ext, active, steps, valid);
}

}  // namespace
}  // namespace aem

namespace aem {
int loglik_f64_soundings(const aem_system *sys, const aem_models_f64 *models, const double *y_obs,
                         int models_per_sounding, const double *eps_an, double eps_mn, double *ll,
                         cudaStream_t stream, const int *active, const int8_t *valid) {
    return launch_forward_f64(sys, models, nullptr, nullptr, y_obs, models_per_sounding, eps_an, eps_mn, ll,
                              (void *)stream, "loglik (SMC, FP64)", active, valid);
}
int loglik_f32_soundings(const aem_system *sys, const aem_models_f32 *models, const double *y_obs,
                         int models_per_sounding, const double *eps_an, double eps_mn, double *ll,
                         cudaStream_t stream, int *counter, const int *active, const int8_t *valid) {
    return launch_forward_f32(sys, models, (float *)nullptr, (float *)nullptr, y_obs, models_per_sounding, eps_an,
                              eps_mn, ll, (void *)stream, "loglik (SMC)", counter, active, nullptr, valid);
}
}  // namespace aem

using namespace aem;

extern "C" int aem_forward_f32(const aem_system *sys, const aem_models_f32 *models, float *gates, float *imh,
                               void *stream) {
    return launch_forward_f32(sys, models, gates, imh, nullptr, 0, nullptr, 0.0, nullptr, stream, "aem_forward_f32");
}

extern "C" int aem_forward_f32_count(const aem_system *sys, const aem_models_f32 *models, float *gates, float *imh,
                                     unsigned long long *layer_steps, void *stream) {
    if (!layer_steps) return fail(AEM_ERR_INVALID_ARG, "aem_forward_f32_count: NULL layer_steps");
    return launch_forward_f32(sys, models, gates, imh, nullptr, 0, nullptr, 0.0, nullptr, stream,
                              "aem_forward_f32_count", nullptr, nullptr, layer_steps);
}

extern "C" int aem_forward_f64(const aem_system *sys, const aem_models_f64 *models, double *gates, double *imh,
                               void *stream) {
    return launch_forward_f64(sys, models, gates, imh, nullptr, 0, nullptr, 0.0, nullptr, stream, "aem_forward_f64");
}

extern "C" int aem_loglik_f32(const aem_system *sys, const aem_models_f32 *models, const double *y_obs,
                              const double *eps_an, double eps_mn, double *ll, float *gates, void *stream) {
    if (!ll && models && models->n_models > 0) return fail(AEM_ERR_INVALID_ARG, "aem_loglik_f32: ll is NULL");
    return launch_forward_f32(sys, models, gates, nullptr, y_obs, 0, eps_an, eps_mn, ll, stream, "aem_loglik_f32");
}

extern "C" int aem_loglik_f64(const aem_system *sys, const aem_models_f64 *models, const double *y_obs,
                              const double *eps_an, double eps_mn, double *ll, double *gates, void *stream) {
    if (!ll && models && models->n_models > 0) return fail(AEM_ERR_INVALID_ARG, "aem_loglik_f64: ll is NULL");
    return launch_forward_f64(sys, models, gates, nullptr, y_obs, 0, eps_an, eps_mn, ll, stream, "aem_loglik_f64");
}

namespace aem {
// Gates and log-likelihood of the FP32 forward model for the adjoint, with the
// per-sounding rows of y_obs (ll may be NULL).
int loglik_gates_f32_soundings(const aem_system *sys, const aem_models_f32 *models, const double *y_obs,
                               int models_per_sounding, const double *eps_an, double eps_mn, double *ll, float *gates,
                               cudaStream_t stream, int *counter, const int8_t *valid) {
    return launch_forward_f32(sys, models, gates, nullptr, y_obs, models_per_sounding, eps_an, eps_mn, ll, stream,
                              "aem_loglik_grad_f32", counter, nullptr, nullptr, valid);
}
}  // namespace aem

extern "C" int aem_system_set_depth_cutoff(aem_system *sys, double attenuation) {
    if (!sys) return fail(AEM_ERR_INVALID_ARG, "aem_system_set_depth_cutoff: NULL system");
    if (!(attenuation >= 0.0) || !(attenuation < 1e30))
        return fail(AEM_ERR_INVALID_ARG, "aem_system_set_depth_cutoff: attenuation must be >= 0 and finite");
    sys->depth_att = (float)attenuation;
    return AEM_OK;
}

extern "C" int aem_autotune_forward(aem_system *sys, const aem_models_f32 *sample, int repeats, void *stream,
                                    int *shape_out, float *ms_out) {
    if (!sys || !sample) return fail(AEM_ERR_INVALID_ARG, "aem_autotune_forward: NULL system or sample");
    if (sample->n_models < 1 || sample->lmax < 1 || sample->lmax > AEM_MAX_LAYERS || repeats < 1)
        return fail(AEM_ERR_INVALID_ARG, "aem_autotune_forward: empty sample, lmax out of range or repeats < 1");
    if (!sample->nlayers || !sample->logsig || !sample->logh || !sample->m || !sample->logtau || !sample->c)
        return fail(AEM_ERR_INVALID_ARG, "aem_autotune_forward: NULL model array");
    cudaStream_t s = (cudaStream_t)stream;
    const int LS = sample->lmax;
    ModelsView<float> mv{sample->n_models, sample->lmax, sample->nlayers, sample->logsig, sample->logh,
                           sample->m, sample->logtau, sample->c};
    float *gates = nullptr;
    AEM_CUDA_TRY(cudaMallocAsync((void **)&gates, sizeof(float) * (size_t)sample->n_models * sys->host.G, s));
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    int rc = AEM_OK, best = -1;
    float best_ms = 0.f;
    if (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess)
        rc = fail(AEM_ERR_CUDA, "aem_autotune_forward: cudaEventCreate");
    for (int c = 0; c < kNumF32Shapes && rc == AEM_OK; ++c) {
        float ms = 0.f;
        // one untimed launch, then the timed repeats
        rc = launch_shape_index(c, sys, mv, LS, gates, nullptr, nullptr, 0, nullptr, 0.0, nullptr, s);
        if (rc == AEM_ERR_UNSUPPORTED) {  // this shape does not fit on an SM: skip it
            rc = AEM_OK;
            if (ms_out) ms_out[c] = -1.f;
            continue;
        }
        if (rc) break;
        cudaEventRecord(e0, s);
        for (int r = 0; r < repeats && rc == AEM_OK; ++r)
            rc = launch_shape_index(c, sys, mv, LS, gates, nullptr, nullptr, 0, nullptr, 0.0, nullptr, s);
        cudaEventRecord(e1, s);
        if (cudaEventSynchronize(e1) != cudaSuccess || cudaEventElapsedTime(&ms, e0, e1) != cudaSuccess) {
            rc = fail(AEM_ERR_CUDA, "aem_autotune_forward: timing");
            break;
        }
        ms /= repeats;
        if (ms_out) ms_out[c] = ms;
        if (best < 0 || ms < best_ms) {
            best = c;
            best_ms = ms;
        }
    }
    if (e0) cudaEventDestroy(e0);
    if (e1) cudaEventDestroy(e1);
    cudaFreeAsync(gates, s);
    if (rc) return rc;
    if (best < 0) return fail(AEM_ERR_UNSUPPORTED, "aem_autotune_forward: no launch shape fits");
    sys->f32_shape[LS] = best;
    if (shape_out) *shape_out = best;
    return AEM_OK;
}

extern "C" int aem_forward_shape(aem_system *sys, int lmax, int shape) {
    if (!sys || lmax < 1 || lmax > AEM_MAX_LAYERS || shape < 0 || shape >= kNumF32Shapes)
        return fail(AEM_ERR_INVALID_ARG, "aem_forward_shape: invalid lmax or shape");
    sys->f32_shape[lmax] = shape;
    return AEM_OK;
}

extern "C" int aem_forward_launch_shape(const aem_system *sys, int lmax, int n_models, int *shape) {
    if (!sys || lmax < 1 || lmax > AEM_MAX_LAYERS || n_models < 0 || !shape)
        return fail(AEM_ERR_INVALID_ARG, "aem_forward_launch_shape: NULL pointer, invalid lmax or n_models < 0");
    return shape_of_launch(sys, lmax, n_models, false, shape);
}
