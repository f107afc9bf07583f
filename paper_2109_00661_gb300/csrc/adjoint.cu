// Gradient of the Gaussian log-likelihood with respect to every merged
// layer's (log10 sigma, log10 h, m, log10 tau, c), by reverse-mode
// differentiation of the forward model (Section 2: Cole-Cole conductivity,
// TE recursion, Hankel sum; Section 2.3.2: gate transform and likelihood).
//
// The FP32 forward kernel (forward.cu) first writes every model's gates and
// log-likelihood.  Then one CTA per model (models claimed from a counter)
// forms the adjoint seeds from those gates,
//   a_f = sum_g T[g,f] dl/dyhat_g,  dl/dyhat = r/v + (e_mn^2 yhat / v)(r^2/v - 1),
// and visits every (frequency, abscissa) item with weight a_f w_k.  Per item,
// bottom-up, with w_n = sqrt(2 (lambda^2 + s_n)) and E_n = exp(-sqrt(2) w_n h_n),
// the down- and upgoing amplitudes (D_n, N_n) at the bottom of every layer n
// follow from the continuity of the field e and of h = w (D - P):
//   D_n, N_n = e +- h / w_n,  P_n = N_n E_n,  e = D_n + P_n,  h = w_n (D_n - P_n)
// from e = 1, h = w of the half-space, up to D_0 = e + h / (sqrt(2) lambda) of
// the air (each interface doubles the scale).  The derivative of R_0 by s_n is
// the integral of the squared field over the layer (the self-adjoint equation's
// sensitivity; its closed form has no interface terms, and between layers only
// the attenuation changes, c_{n+1} = 4 E_n c_n):
//   dR_0/ds_n = -c_n [(1 - E_n)(D_n^2 + N_n P_n) 2 / w_n + 4 sqrt(2) h_n D_n P_n],
//   dR_0/dh_n = -c_n sqrt(2) w_n^2 4 D_n P_n,  c_0 = 1 / (D_0^2 sqrt(2) lambda),
//   dR_0/ds = -c 2 / w for the half-space.
// For each layer Im(dR_0/ds_n ds_n/dp) and Im(dR_0/dh_n) go into per-thread
// accumulators, reduced over the CTA at the end of the model.  R_0 is
// holomorphic in every s_n, so d Im R_0 / dp = Im(dR_0/ds_n ds_n/dp) for the
// real parameters p.
//
// Like the forward kernel, each thread carries two abscissae of one frequency
// (k and k + K/2) through both passes in 64-bit register pairs on the paired
// FP32 instructions (f32x2.h); the two abscissae's weighted adjoints are added
// before they meet the per-(frequency, layer) derivatives ds_n/dp, which do
// not depend on the abscissa.
//
// The bound is the instruction issue of the paired FP32 and special-function
// units: about 100 paired operations and 20 special-function ones per pair and
// layer for both passes.  Differentiating the Moebius chain interface by
// interface took 163 and 28: 16384 models of 60 x 200 items with 1 to 10
// layers, forward kernel included, 7.05 -> 4.86 ms.  E_n is formed again on the
// way down: kept from the way up it costs 16 bytes of local memory per layer
// each way, 5.58 against 5.23 ms.
#include <cuda_runtime.h>

#include <cstdint>
#include <type_traits>

#include "aem_internal.h"
#include "depth_cutoff.h"
#include "f32x2.h"
#include "te_roots.h"

namespace aem {
namespace {

using namespace f32x2;

constexpr int kGT = 256;
constexpr int kGW = kGT / 32;
constexpr int kNP = 5;  // parameters per layer: log10 sigma, log10 h, m, log10 tau, c
constexpr unsigned kMask = 0xffffffffu;

// scalar complex helpers of the per-(frequency, layer) Cole-Cole setup
__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
    return make_float2(fmaf(a.x, b.x, -a.y * b.y), fmaf(a.x, b.y, a.y * b.x));
}
__device__ __forceinline__ float2 cscale(float2 a, float s) { return make_float2(a.x * s, a.y * s); }
__device__ __forceinline__ float2 crcp(float2 a) {
    const float d = 1.0f / fmaf(a.x, a.x, a.y * a.y);
    return make_float2(a.x * d, -a.y * d);
}

// paired complex helpers: two abscissae per operation
__device__ __forceinline__ C2x2 c2(u64 re, u64 im) {
    C2x2 r;
    r.re = re;
    r.im = im;
    return r;
}
__device__ __forceinline__ C2x2 c2mul(C2x2 a, C2x2 b) {
    return c2(sub2(mul2(a.re, b.re), mul2(a.im, b.im)), fma2(a.re, b.im, mul2(a.im, b.re)));
}
__device__ __forceinline__ C2x2 c2mulc(C2x2 a, C2x2 b) {  // a conj(b)
    return c2(fma2(a.re, b.re, mul2(a.im, b.im)), sub2(mul2(a.im, b.re), mul2(a.re, b.im)));
}
__device__ __forceinline__ C2x2 c2sq(C2x2 a) {
    const u64 t = mul2(a.re, a.im);
    return c2(mul2(sub2(a.re, a.im), add2(a.re, a.im)), add2(t, t));
}
// The power of two next to 1 / max(|Re d|, |Im d|), per abscissa (2^-126 .. 2^126;
// of zero, an infinity or a NaN one of the ends).
__device__ __forceinline__ float pow2_inv(float a, float b) {
    const int e = __float_as_int(fmaxf(fabsf(a), fabsf(b))) >> 23;
    return __int_as_float(min(max(254 - e, 1), 253) << 23);
}
__device__ __forceinline__ u64 pow2_inv2(C2x2 d) {
    float a0, a1, b0, b1;
    up2(d.re, a0, a1);
    up2(d.im, b0, b1);
    return pk2(pow2_inv(a0, b0), pow2_inv(a1, b1));
}
constexpr u64 kTwo2 = 0x4000000040000000ull, kQuarter2 = 0x3e8000003e800000ull;
constexpr u64 kMinusHalf2 = 0xbf000000bf000000ull, kMinusOne2 = 0xbf800000bf800000ull;

// root2 and 1 / m (for dw/ds = 1 / w = conj(w) / (2 m)).
__device__ __forceinline__ Root root2_inv(u64 lam2, ulonglong2 rec, u64 &inv_m) {
    const u64 x = add2(lam2, rec.x);
    const u64 v = fma2(x, x, mul2(rec.y, rec.y));
    float v0, v1, x0, x1;
    up2(v, v0, v1);
    up2(x, x0, x1);
    inv_m = pk2(rsqrt_approx(v0), rsqrt_approx(v1));
    Root w;
    w.m = mul2(v, inv_m);
    float m0, m1;
    up2(w.m, m0, m1);
    const float t0 = m0 + fabsf(x0), t1 = m1 + fabsf(x1);
    const u64 rr = pk2(rsqrt_approx(t0), rsqrt_approx(t1));
    float p0, p1, o0, o1;
    up2(mul2(pk2(t0, t1), rr), p0, p1);
    up2(mul2(rec.y, rr), o0, o1);
    w.re = pk2(x0 >= 0.f ? p0 : o0, x1 >= 0.f ? p1 : o1);
    w.im = pk2(x0 >= 0.f ? o0 : p0, x1 >= 0.f ? o1 : p1);
    return w;
}

// E = exp(-sqrt(2) w h) for both abscissae (FOUR: 4 E); he = (e x 2, e ln2 x 2), e = -sqrt(2) h log2 e
template <bool FOUR>
__device__ __forceinline__ C2x2 c2expm(ulonglong2 he, const Root &w) {
    float a0, a1, f0, f1, s0, c0, s1, c1;
    up2(FOUR ? fma2(he.x, w.re, kTwo2) : mul2(he.x, w.re), a0, a1);
    up2(reduce_2pi2(mul2(he.y, w.im)), f0, f1);
    sincos_approx(f0, &s0, &c0);
    sincos_approx(f1, &s1, &c1);
    const u64 e = pk2(ex2_approx(a0), ex2_approx(a1));
    return c2(mul2(e, pk2(c0, c1)), mul2(e, pk2(s0, s1)));
}

template <class T>
__device__ __forceinline__ T wsum(T v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kMask, v, o);
    return v;
}

struct GradModels {
    int n, lmax;
    const int8_t *nlayers;
    const float *logsig, *logh, *m, *logtau, *c;
};

// Shared memory (dynamic), in order: RS[F*LS] (ulonglong2: (Re s, Re s),
// (Im s, Im s)), lamp[K2] (ulonglong2: (lam_a^2, lam_b^2), 1 / (sqrt(2) lambda)),
// DS[F*LS*2] (float4: ds/dp for log10 sigma and m, then for log10 tau and c),
// hwp[K2] (float2 weights of the pair over sqrt(2) lambda), af[F], T[G*F],
// part[kGW * LS * kNP], TH[F*LS] (float: the depth cutoff's thresholds).
size_t grad_smem_bytes(int F, int G, int K, int LS) {
    const size_t K2 = (size_t)(K + 1) / 2, FL = (size_t)F * LS;
    return sizeof(ulonglong2) * (FL + K2) + sizeof(float4) * (FL * 2) + sizeof(float2) * K2 +
           sizeof(float) * ((size_t)F + (size_t)G * F + (size_t)kGW * LS * kNP + FL);
}

// MAXL: the largest layer count the per-thread arrays hold (10 or
// AEM_MAX_LAYERS), so the common lmax <= 10 keeps them half as large.  Three
// resident CTAs per SM (80 registers) measure faster than two (120 registers,
// 5.9 against 5.2 ms of the workload above) and like four (64, spilling).
template <int MAXL>
__global__ void __launch_bounds__(kGT, 3) loglik_grad_kernel(GradModels mv, int F, int G, int K, int LS, int cc_form,
                                                             float len,
                                                             const float *__restrict__ g_omega,
                                                             const float *__restrict__ g_lam,
                                                             const float *__restrict__ g_hw,
                                                             const float *__restrict__ g_T,
                                                             const double *__restrict__ y_obs, int obs_per,
                                                             const double *__restrict__ eps_an, double eps_mn,
                                                             const float *__restrict__ g_gates, float *__restrict__ grad,
                                                             int *__restrict__ work_counter, float att0,
                                                             const int8_t *__restrict__ valid) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int K2 = (K + 1) / 2;
    const size_t FL = (size_t)F * LS;
    ulonglong2 *RS = reinterpret_cast<ulonglong2 *>(smem_raw);
    ulonglong2 *lamp = RS + FL;
    float4 *DS = reinterpret_cast<float4 *>(lamp + K2);
    float2 *hwp = reinterpret_cast<float2 *>(DS + FL * 2);
    float *af = reinterpret_cast<float *>(hwp + K2);
    float *Ts = af + F;
    float *part = Ts + (size_t)G * F;
    float *TH = part + (size_t)kGW * LS * kNP;
    __shared__ ulonglong2 HE[AEM_MAX_LAYERS];
    __shared__ float thick[AEM_MAX_LAYERS];
    __shared__ float sig_s[AEM_MAX_LAYERS], m_s[AEM_MAX_LAYERS], tau_s[AEM_MAX_LAYERS], c_s[AEM_MAX_LAYERS];
    __shared__ double dldy[AEM_MAX_GATES];

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // lengths in the forward kernel's unit (aem_system::len)
    const float mu0 = (float)kMu0 * len * len, ilen = 1.f / len, ln10 = 2.302585092994046f;
    for (int i = tid; i < G * F; i += blockDim.x) Ts[i] = g_T[i];
    // abscissa pairs (k, k + K2); an odd K pads the last pair with a zero weight
    for (int k = tid; k < K2; k += blockDim.x) {
        const int kb = k + K2 < K ? k + K2 : K - 1;
        const float la = g_lam[k], lb = g_lam[kb];
        lamp[k] = make_ulonglong2(pk2(la * la, lb * lb), pk2(0.70710678118654752f / la, 0.70710678118654752f / lb));
        hwp[k] = make_float2(0.70710678118654752f / la * g_hw[k],
                             k + K2 < K ? 0.70710678118654752f / lb * g_hw[kb] : 0.f);
    }
    const int FK2 = F * K2;

    // models are claimed from a counter as CTAs finish them (model costs vary
    // with the layer count, so a fixed stride would leave SMs idle at the end)
    __shared__ int next_model;
    for (int p = blockIdx.x; p < mv.n; p = next_model) {
        const int L = mv.nlayers[p];
        __syncthreads();
        // when this model's items are done, not before (forward.cu)
        auto ask = [&] {
            if (tid == 0) next_model = (int)gridDim.x + atomicAdd(work_counter, 1);
        };
        if (valid && !valid[p]) {  // a proposal the caller will not use (CTA-uniform)
            ask();
            __syncthreads();  // next_model visible to every thread
            continue;
        }
        if (tid < L) {
            const size_t o = (size_t)p * mv.lmax + tid;
            sig_s[tid] = exp10f(mv.logsig[o]);
            const float h = exp10f(mv.logh[o]) * ilen;
            thick[tid] = h;
            const float e = -1.41421356237309505f * 1.44269504088896341f * h;
            HE[tid] = make_ulonglong2(pk2(e, e), pk2(e * 0.69314718055994531f, e * 0.69314718055994531f));
            m_s[tid] = mv.m[o];
            tau_s[tid] = exp10f(mv.logtau[o]);
            c_s[tid] = mv.c[o];
        }
        __syncthreads();
        // Cole-Cole and its derivatives, per (frequency, layer), with
        // x = (w tau)^c e^{i pi c / 2} and s = i w mu0 sig:
        //   paper   sig = s_inf (1 - m / (1 + x))
        //   Pelton  sig = s_0 (1 + x) / (1 + (1 - m) x)
        //   literal sig = s_0 (1 + (1 - m) x) / (1 + x)
        for (int i = tid; i < F * L; i += blockDim.x) {
            const int f = i / L, n = i - f * L;
            const float w = g_omega[f];
            const float si = sig_s[n], mm = m_s[n], cc = c_s[n];
            const float lwt = logf(w * tau_s[n]);
            const float mag = expf(cc * lwt);
            float sp, cp;
            sincospif(0.5f * cc, &sp, &cp);
            const float2 x = make_float2(mag * cp, mag * sp);
            const float2 ix1 = crcp(make_float2(1.f + x.x, x.y));  // 1 / (1 + x)
            float2 sg, dsg_dm, dsg_dx;
            // sig itself without cancellation, as the forward kernel forms it:
            // real parts as sums of non-negative terms (Re x >= 0), imaginary
            // parts as the single product m Im x / |.|^2
            if (cc_form == AEM_CC_PAPER) {
                // s_inf ((1 - m) + x) / (1 + x); ix1.y <= 0
                sg = make_float2(si * fmaf((1.f - mm) + x.x, ix1.x, -x.y * ix1.y), -si * mm * ix1.y);
                dsg_dm = cscale(ix1, -si);
                dsg_dx = cscale(cmul(ix1, ix1), si * mm);                // s_inf m / (1 + x)^2
            } else {
                const float2 b = make_float2(1.f + (1.f - mm) * x.x, (1.f - mm) * x.y);  // 1 + (1 - m) x
                if (cc_form == AEM_CC_PELTON) {
                    const float2 ib = crcp(b);                           // conj(b) / |b|^2
                    sg = make_float2(si * fmaf(1.f + x.x, ib.x, -x.y * ib.y), si * mm * x.y / (b.x * b.x + b.y * b.y));
                    dsg_dm = cmul(sg, cmul(x, ib));                      // sig x / (1 + (1 - m) x)
                    dsg_dx = cscale(cmul(ib, ib), si * mm);              // s_0 m / (1 + (1 - m) x)^2
                } else {
                    sg = make_float2(si * fmaf(b.x, ix1.x, -b.y * ix1.y), si * mm * ix1.y);
                    dsg_dm = cscale(cmul(x, ix1), -si);                  // -s_0 x / (1 + x)
                    dsg_dx = cscale(cmul(ix1, ix1), -si * mm);           // -s_0 m / (1 + x)^2
                }
            }
            const float2 dx_dlt = cscale(x, cc * ln10);                   // d x / d log10 tau
            const float2 dx_dc = cmul(x, make_float2(lwt, 1.57079632679489662f));
            const float2 iwm = make_float2(0.f, w * mu0);                 // i w mu0
            const float2 sv = cmul(iwm, sg);
            RS[(size_t)f * LS + n] = make_ulonglong2(pk2(sv.x, sv.x), pk2(sv.y, sv.y));
            const float2 d0 = cmul(iwm, cscale(sg, ln10)), d1 = cmul(iwm, dsg_dm);
            const float2 d2 = cmul(iwm, cmul(dsg_dx, dx_dlt)), d3 = cmul(iwm, cmul(dsg_dx, dx_dc));
            float4 *d = DS + ((size_t)f * LS + n) * 2;
            d[0] = make_float4(d0.x, d0.y, d1.x, d1.y);
            d[1] = make_float4(d2.x, d2.y, d3.x, d3.y);
        }
        __syncthreads();

        // ---- the depth cutoff's thresholds (depth_cutoff.h), one frequency per
        // thread; each item then runs only the layers its abscissa needs (the
        // forward kernel runs at least those: the largest count of the item's
        // 32-item group), so a layer it drops contributes nothing to this
        // item's gradient, a change under exp(-att0) of the item's share
        const bool cut = att0 > 0.f && L > 1;
        if (cut)
            for (int f = tid; f < F; f += blockDim.x)
                depth_thresholds(
                    [&](int n) {
                        float sx, sy, t;
                        up2(RS[(size_t)f * LS + n].x, sx, t);
                        up2(RS[(size_t)f * LS + n].y, sy, t);
                        return make_float2(sx, sy);
                    },
                    thick, L, att0, TH + (size_t)f * LS);
        // ---- dl/dyhat from the forward kernel's gates of this model
        if (tid < G) {
            const double yh = (double)g_gates[(size_t)p * G + tid];
            const double ea = eps_an[tid];
            const double v = ea * ea + (eps_mn * yh) * (eps_mn * yh);
            const double r = y_obs[(size_t)(p / obs_per) * G + tid] - yh;
            dldy[tid] = r / v + (eps_mn * eps_mn * yh / v) * (r * r / v - 1.0);
        }
        __syncthreads();
        for (int j = tid; j < F; j += blockDim.x) {
            double a = 0.0;
            for (int g = 0; g < G; ++g) a += (double)Ts[g * F + j] * dldy[g];
            af[j] = (float)a;
        }
        __syncthreads();

        // ---- reverse sweep per pair of items, per-thread accumulators (one
        // 16-byte access for the four that come together); acc_h holds the sum
        // of Im(c 4 D P (lambda^2 + s)) until the reduction applies
        // -2 sqrt(2) h_n ln10
        float4 acc_s[MAXL];
        float acc_h[MAXL];
        for (int v = 0; v < L; ++v) {
            acc_s[v] = make_float4(0.f, 0.f, 0.f, 0.f);
            acc_h[v] = 0.f;
        }
        C2x2 Ns[MAXL], Ds[MAXL];
        u64 Sc[MAXL];  // the powers of two of the scaled sweep
        int f = tid / K2, k = tid - (tid / K2) * K2;
        for (int item = tid; item < FK2; item += blockDim.x) {
            const ulonglong2 lp = lamp[k];  // (lam^2 pair, 1 / (sqrt(2) lam) pair)
            const ulonglong2 *Sf = RS + (size_t)f * LS;
            const float4 *Df = DS + (size_t)f * LS * 2;
            int Li = L;  // the layers this item runs
            if (cut) {
                float l2, lb2;
                up2(lp.x, l2, lb2);
                Li = depth_layers(l2, TH + (size_t)f * LS, L);
            }
            auto emit = [&](int n, C2x2 t) {
                float x0, x1, y0, y1;
                up2(t.re, x0, x1);
                up2(t.im, y0, y1);
                const float swx = x0 + x1, swy = y0 + y1;
                const float4 d01 = Df[2 * n], d23 = Df[2 * n + 1];
                float4 ac = acc_s[n];
                ac.x += fmaf(swx, d01.y, swy * d01.x);
                ac.y += fmaf(swx, d01.w, swy * d01.z);
                ac.z += fmaf(swx, d23.y, swy * d23.x);
                ac.w += fmaf(swx, d23.w, swy * d23.z);
                acc_s[n] = ac;
            };
            // false: D_0 has left the range in which the squares of every
            // layer's amplitudes stay normal FP32 numbers, and nothing was
            // added: many thick layers of alternating contrast, where each
            // interface multiplies D by up to the contrast of w.  The scaled
            // sweep then brings every (N_n, D_n) back to about one by a power
            // of two; done always, it costs 5 %.
            auto sweep = [&](auto sc) -> bool {
                constexpr bool SCALED = decltype(sc)::value;
                // bottom-up
                u64 im;
                Root w = root2_inv(lp.x, Sf[Li - 1], im);
                C2x2 e = c2(kOne2, kZero2), h = c2(w.re, w.im);
                for (int n = Li - 2; n >= 0; --n) {
                    w = root2_inv(lp.x, Sf[n], im);
                    const C2x2 g = c2mulc(h, c2(mul2(w.re, im), mul2(w.im, im)));
                    C2x2 N = c2(fma2(kMinusHalf2, g.re, e.re), fma2(kMinusHalf2, g.im, e.im));
                    C2x2 D = c2(fma2(kHalf2, g.re, e.re), fma2(kHalf2, g.im, e.im));
                    if constexpr (SCALED) {
                        const u64 q = pow2_inv2(D);
                        N = c2(mul2(N.re, q), mul2(N.im, q));
                        D = c2(mul2(D.re, q), mul2(D.im, q));
                        Sc[n] = q;
                    }
                    Ns[n] = N;
                    Ds[n] = D;
                    const C2x2 P = c2mul(N, c2expm<false>(HE[n], w));
                    e = c2(add2(D.re, P.re), add2(D.im, P.im));
                    h = c2mul(c2(w.re, w.im), c2(sub2(D.re, P.re), sub2(D.im, P.im)));
                }
                const C2x2 D0 = c2(fma2(h.re, lp.y, e.re), fma2(h.im, lp.y, e.im));
                float d0, d1;
                up2(fma2(D0.re, D0.re, mul2(D0.im, D0.im)), d0, d1);
                if (!SCALED && !(d0 > 1e-24f && d1 > 1e-24f && d0 < 1e30f && d1 < 1e30f)) return false;
                const float2 hw = hwp[k];
                const float a = af[f];
                const u64 i = pk2(rcp_approx(d0), rcp_approx(d1)), wgt = pk2(a * hw.x, a * hw.y);
                C2x2 c = c2sq(c2(mul2(D0.re, i), sub2(kZero2, mul2(D0.im, i))));
                c = c2(mul2(c.re, wgt), mul2(c.im, wgt));
                // top-down
                for (int n = 0; n < Li - 1; ++n) {
                    const ulonglong2 he = HE[n], sv = Sf[n];
                    w = root2_inv(lp.x, sv, im);
                    const C2x2 E4 = c2expm<true>(he, w), N = Ns[n], D = Ds[n];
                    const C2x2 P4 = c2mul(N, E4), D2 = c2sq(D), NP4 = c2mul(N, P4), T4 = c2mul(D, P4);
                    // -(1 - E) (D^2 + N P) 2 / w - sqrt(2) h 4 T
                    C2x2 A = c2mul(c2(fma2(NP4.re, kQuarter2, D2.re), fma2(NP4.im, kQuarter2, D2.im)),
                                   c2(fma2(E4.re, kQuarter2, kMinusOne2), mul2(E4.im, kQuarter2)));
                    A = c2mulc(A, c2(mul2(w.re, im), mul2(w.im, im)));
                    A = c2(fma2(he.y, T4.re, A.re), fma2(he.y, T4.im, A.im));
                    emit(n, c2mul(c, A));
                    const C2x2 cT = c2mul(c, T4);
                    float h0, h1;
                    up2(fma2(cT.im, add2(lp.x, sv.x), mul2(cT.re, sv.y)), h0, h1);
                    acc_h[n] += h0 + h1;
                    c = c2mul(c, E4);
                    if constexpr (SCALED) {
                        const u64 q = mul2(Sc[n], Sc[n]);
                        c = c2(mul2(c.re, q), mul2(c.im, q));
                    }
                }
                w = root2_inv(lp.x, Sf[Li - 1], im);
                const u64 ni = sub2(kZero2, im);
                emit(Li - 1, c2mulc(c, c2(mul2(w.re, ni), mul2(w.im, ni))));
                return true;
            };
            if (!sweep(std::false_type{})) sweep(std::true_type{});
            k += blockDim.x;
            while (k >= K2) {
                k -= K2;
                ++f;
            }
        }
        ask();
        // CTA reduction of the per-thread accumulators (fixed order)
        for (int n = 0; n < L; ++n) {
            const float4 ac = acc_s[n];
            const float s0 = wsum<float>(ac.x), s1 = wsum<float>(acc_h[n]), s2 = wsum<float>(ac.y),
                        s3 = wsum<float>(ac.z), s4 = wsum<float>(ac.w);
            if (lane == 0) {
                float *q = part + (warp * LS + n) * kNP;
                q[0] = s0;
                q[1] = s1;
                q[2] = s2;
                q[3] = s3;
                q[4] = s4;
            }
        }
        __syncthreads();
        for (int v = tid; v < mv.lmax * kNP; v += blockDim.x) {
            float s = 0.f;
            if (v < L * kNP) {
                for (int w = 0; w < kGW; ++w) s += part[w * LS * kNP + v];
                if (v % kNP == 1) s *= -2.f * 1.41421356237309505f * thick[v / kNP] * ln10;
            }
            grad[(size_t)p * mv.lmax * kNP + v] = s;
        }
    }
}

}  // namespace
}  // namespace aem

using namespace aem;

namespace aem {

// scratch layout: the adjoint kernel's claim counter at 0, the forward
// kernel's at 64, the gates [P][G] from 256
constexpr size_t kGateOff = 256;
size_t grad_work_bytes(int n_models, int G) { return kGateOff + sizeof(float) * (size_t)n_models * G; }

int loglik_grad_f32_soundings(const aem_system *sys, const aem_models_f32 *models, const double *y_obs,
                              int models_per_sounding, const double *eps_an, double eps_mn, double *ll, float *grad,
                              cudaStream_t stream, void *work_ext, const int8_t *valid) {
    const SystemTables &h = sys->host;
    const int LS = models->lmax;
    const size_t smem = grad_smem_bytes(h.F, h.G, h.K, LS);
    auto kern = LS <= 10 ? loglik_grad_kernel<10> : loglik_grad_kernel<AEM_MAX_LAYERS>;
    int per_sm = 0;
    if (const int rc = resident_ctas(&sys->grad_ctas[LS], kern, kGT, smem, sys->device, &per_sm)) return rc;
    if (per_sm < 1) per_sm = 1;
    long long grid = (long long)sys->num_sms * per_sm;
    if (grid > models->n_models) grid = models->n_models;
    GradModels gm{models->n_models, models->lmax, models->nlayers, models->logsig, models->logh,
                  models->m, models->logtau, models->c};
    void *work = work_ext;
    if (!work_ext) AEM_CUDA_TRY(cudaMallocAsync(&work, grad_work_bytes(models->n_models, h.G), stream));
    int *counter = static_cast<int *>(work);
    int *fwd_counter = reinterpret_cast<int *>(static_cast<char *>(work) + 64);
    float *gates = reinterpret_cast<float *>(static_cast<char *>(work) + kGateOff);
    int rc = loglik_gates_f32_soundings(sys, models, y_obs, models_per_sounding, eps_an, eps_mn, ll, gates, stream,
                                        fwd_counter, valid);
    cudaError_t e = cudaSuccess;
    if (rc == AEM_OK) {
        e = cudaMemsetAsync(counter, 0, sizeof(int), stream);
        if (e == cudaSuccess) {
            kern<<<(unsigned)grid, kGT, smem, stream>>>(gm, h.F, h.G, h.K, LS, h.cc_form, sys->len, sys->d_omega_f,
                                                        sys->d_lamu_f, sys->d_hw_f, sys->d_T_f, y_obs, models_per_sounding, eps_an,
                                                        eps_mn, gates, grad, counter, sys->depth_att, valid);
            e = cudaGetLastError();
        }
    }
    if (!work_ext) cudaFreeAsync(work, stream);
    if (rc) return rc;
    AEM_CUDA_TRY(e);
    return AEM_OK;
}

}  // namespace aem

extern "C" int aem_loglik_grad_f32(const aem_system *sys, const aem_models_f32 *models, const double *y_obs,
                                   const double *eps_an, double eps_mn, double *ll, float *grad, void *stream) {
    if (!sys || !models) return fail(AEM_ERR_INVALID_ARG, "aem_loglik_grad_f32: NULL system or models");
    if (models->n_models < 0 || models->lmax < 1 || models->lmax > AEM_MAX_LAYERS)
        return fail(AEM_ERR_INVALID_ARG, "aem_loglik_grad_f32: n_models < 0 or lmax outside 1..AEM_MAX_LAYERS");
    if (models->n_models == 0) return AEM_OK;
    if (!grad || !y_obs || !eps_an || !models->nlayers || !models->logsig || !models->logh || !models->m ||
        !models->logtau || !models->c)
        return fail(AEM_ERR_INVALID_ARG, "aem_loglik_grad_f32: NULL pointer");
    return loglik_grad_f32_soundings(sys, models, y_obs, models->n_models, eps_an, eps_mn, ll, grad,
                                     (cudaStream_t)stream);
}
