// Gate transform y = T Im H (Section 2.3.2: step-off gates from the
// frequency-domain response) and the Gaussian log-likelihood, from a batch of
// spectra, on the 5th-generation tensor cores.
//
// The transform is the one dense contraction of the path: D[P x G] =
// A[P x F] B[G x F]^T with A the spectra and B the transform matrix.  The
// spectra are FP32 and the transform is ill-conditioned (terms of both signs
// cancel), so each operand is split into a high and a low part in the tensor
// input type and three products are accumulated in FP32:
//   D = A_hi B_hi + A_hi B_lo + A_lo B_hi
// (the dropped A_lo B_lo term is below the split's own rounding).  TF32
// (11-bit significand) leaves a relative residual near 2^-22 per term, BF16
// (8-bit) near 2^-17.
//
// One CTA of eight warps per 128-model tile (persistent over tiles, several
// CTAs per SM so that one CTA's staging overlaps another's MMA and epilogue):
// the threads stage A_hi / A_lo of the tile and, once per CTA, B_hi / B_lo in
// shared memory in the canonical K-major layout without swizzle (core
// matrices of 8 rows x 16 bytes), each lane converting one 16-byte core-matrix
// row so that a warp's stores cover 512 contiguous bytes; one thread issues
// the tcgen05.mma chain into one of two TMEM accumulators (row m of the tile
// in TMEM lane m, gate n in column n) and commits it to an mbarrier; while the
// next tile's chain runs into the other one, every warp reads its 32 lanes
// (warps w and w + 4 the same lanes, each half of the columns) with tcgen05.ld
// and forms the gates and the likelihood terms of its 32 models, the two
// halves' sums meeting in shared memory.  The likelihood terms are FP32
// (Section 2.3.2's Gaussian: the residual from a float pair holding the FP64
// datum, the variance, a division, and the logarithm of a product of variances,
// see LlAcc) and their sum is carried as an unevaluated FP32 pair (Knuth's
// TwoSum), so no FP64 arithmetic is left per gate.  Every wait is bounded:
// on a timeout the CTA records AEM_ERR_TIMEOUT in the system's status word,
// waits (bounded) once more for its own MMAs, frees its TMEM and returns.  If
// that second wait also gives up, the MMAs it issued may still be in flight
// when the TMEM is freed, which the tcgen05 model leaves undefined: the
// recorded timeout then means the device context should be treated as
// unreliable.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cstdint>
#include <type_traits>

#include "aem_internal.h"
#include "f32x2.h"

namespace aem {
namespace {

using f32x2::two_sum;

constexpr int kTM = 128;       // models per tile = MMA M
constexpr int kThreads = 256;  // warps w and w + 4 read TMEM lanes 32 (w mod 4) .., one half of the columns each
constexpr uint32_t kSpinLimit = 1u << 22;
constexpr double kLn2Pi = 1.83787706640934548356;  // ln(2 pi)

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

// Shared-memory matrix descriptor (no swizzle): start address, leading
// (K-direction core matrix) byte offset and stride (8-row group) byte offset in
// 16-byte units at bits 0-13, 16-29 and 32-45; descriptor version 1 at bit 46;
// base offset 0, swizzle mode 0.
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr, uint32_t lbo, uint32_t sbo) {
    return (uint64_t)((addr >> 4) & 0x3FFFu) | ((uint64_t)((lbo >> 4) & 0x3FFFu) << 16) |
           ((uint64_t)((sbo >> 4) & 0x3FFFu) << 32) | (1ull << 46);
}

// Instruction descriptor for kind::tf32 / kind::f16: FP32 accumulator (bits
// 4-5 = 1), A and B formats at bits 7-9 and 10-12 (BF16 = 1, TF32 = 2), both
// operands K-major (bits 15, 16 = 0), N >> 3 at bits 17-22, M >> 4 at 24-28.
__host__ __device__ constexpr uint32_t instr_desc(uint32_t fmt, uint32_t M, uint32_t N) {
    return (1u << 4) | (fmt << 7) | (fmt << 10) | ((N >> 3) << 17) | ((M >> 4) << 24);
}

template <int KIND>  // 0: TF32 split, 1: BF16 split
__device__ __forceinline__ void mma(uint32_t d_tmem, uint64_t da, uint64_t db, uint32_t idesc, uint32_t accumulate) {
    if constexpr (KIND == 0) {
        asm volatile(
            "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
            "tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(d_tmem),
            "l"(da), "l"(db), "r"(idesc), "r"(accumulate));
    } else {
        asm volatile(
            "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
            "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(d_tmem),
            "l"(da), "l"(db), "r"(idesc), "r"(accumulate));
    }
}

__device__ __forceinline__ void mma_commit(uint32_t mbar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(mbar)
                 : "memory");
}

__device__ __forceinline__ void mbar_init(uint32_t mbar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(mbar), "r"(count) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint32_t mbar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}\n"
        : "=r"(ok)
        : "r"(mbar), "r"(parity)
        : "memory");
    return ok != 0;
}

// Bounded wait for the given phase parity of the mbarrier.
__device__ __forceinline__ bool mbar_wait_bounded(uint32_t mbar, uint32_t parity, uint32_t limit = kSpinLimit) {
    for (uint32_t i = 0; i < limit; ++i)
        if (mbar_try_wait(mbar, parity)) return true;
    return false;
}

__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void tc_before_sync() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_after_sync() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

__device__ __forceinline__ void tmem_alloc(uint32_t slot, uint32_t ncols) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(slot), "r"(ncols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}

__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}

// Eight consecutive FP32 columns of this thread's TMEM lane; the wait takes
// the registers as operands so that no use is scheduled before it.
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, float v[8]) {
    uint32_t r0, r1, r2, r3, r4, r5, r6, r7;
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3), "=r"(r4), "=r"(r5), "=r"(r6), "=r"(r7)
                 : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(r0), "+r"(r1), "+r"(r2), "+r"(r3), "+r"(r4), "+r"(r5), "+r"(r6), "+r"(r7)::"memory");
    v[0] = __uint_as_float(r0);
    v[1] = __uint_as_float(r1);
    v[2] = __uint_as_float(r2);
    v[3] = __uint_as_float(r3);
    v[4] = __uint_as_float(r4);
    v[5] = __uint_as_float(r5);
    v[6] = __uint_as_float(r6);
    v[7] = __uint_as_float(r7);
}

// High / low split of x in the tensor input type (raw bits).
template <int KIND>
struct Split;
template <>
struct Split<0> {
    using T = uint32_t;
    static constexpr int ES = 4;
    __device__ static void run(float x, uint32_t &hi, uint32_t &lo) {
        asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(hi) : "f"(x));
        const float r = x - __uint_as_float(hi);
        asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(lo) : "f"(r));
    }
    // The same for finite x in integers: round to 11 bits, ties away, by adding
    // half of the 13 dropped ones (the conversion takes some four instructions).
    // The tensor core ignores an operand's low 13 bits, so lo needs no mask.  A
    // NaN's bits would carry out of the format: the caller converts those above.
    __device__ static void run_finite(float x, uint32_t &hi, uint32_t &lo) {
        hi = (__float_as_uint(x) + 0x1000u) & 0xffffe000u;
        lo = __float_as_uint(x - __uint_as_float(hi)) + 0x1000u;
    }
    static constexpr float kFinite = 1.7e38f;  // half of the largest, so that hi stays finite
};
template <>
struct Split<1> {
    using T = uint16_t;
    static constexpr int ES = 2;
    __device__ static void run(float x, uint16_t &hi, uint16_t &lo) {
        const __nv_bfloat16 h = __float2bfloat16_rn(x);
        const __nv_bfloat16 l = __float2bfloat16_rn(x - __bfloat162float(h));
        hi = __bfloat16_as_ushort(h);
        lo = __bfloat16_as_ushort(l);
    }
    __device__ static void run_finite(float x, uint16_t &hi, uint16_t &lo) { run(x, hi, lo); }
    static constexpr float kFinite = 1.7e38f;
};

struct TcArgs {
    const float *imh;  // [P][F]
    int P, F, G, KP, N, ncols;
    const float *T;  // [G][F]
    const double *y_obs;
    int obs_per;
    const double *eps_an;
    double eps_mn;
    float *gates;  // [P][G] or null
    double *ll;    // [P] or null
    int *status;
    float gh, gl;    // G ln 2 pi as a float pair
    uint32_t spins;  // iteration limit of the completion wait
    int skip_mma;    // diagnostics: issue nothing for the first tile (the wait then runs out)
};

// The likelihood terms of one model's gates (Section 2.3.2): for gate g, yh
// the prediction, (yhi, ylo) the float pair of the datum and ea2 = eps_an^2,
//   r = (yhi - yh) + ylo,  v = ea2 + (eps_mn yh)^2,
// and ll = -1/2 (sum r^2 / v + sum ln v + G ln 2 pi), formed in FP64 once per
// model.  The quotients are FP32, rounded once (a reciprocal and one residual
// step), their sum an unevaluated FP32 pair (TwoSum).  The logarithms need none
// per gate: v = m 2^e, the m in [1, 2) multiply up (a factor 2^-24 each) and the
// e add up exactly, and sum ln v = ln2 sum e + ln prod m (a single-precision
// ln v near -45 rounds by 2e-6, the product's factor by 6e-8).  No branch per
// gate, so that the gates overlap: a library division and logarithm each made
// the epilogue a chain of some 2,500 cycles per tile.  A quotient or variance
// outside the range this is exact in marks the model, and the caller forms its
// terms again with `exact` (the library's functions).
struct LlAcc {
    float s = 0.f, e = 0.f, prod = 1.f;
    int ex = 0;
    bool odd = false;
    __device__ __forceinline__ void plus(float t) {
        float s1, e1;
        two_sum(s, t, s1, e1);
        s = s1;
        e += e1;
    }
    template <bool EXACT>
    __device__ __forceinline__ void add(float yh, float2 y, float ea2, float em) {
        const float r = (y.x - yh) + y.y;
        const float q = em * yh;
        const float v = fmaf(q, q, ea2);
        const float r2 = r * r;
        if constexpr (EXACT) {
            plus(__fdiv_rn(r2, v) + logf(v));
        } else {
            const unsigned bits = __float_as_uint(v);
            float i;
            asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(i) : "f"(v));
            float t = r2 * i;
            t = fmaf(fmaf(-t, v, r2), i, t);
            plus(t);
            ex += (int)(bits >> 23) - 127;
            prod *= __uint_as_float((bits & 0x7fffffu) | 0x3f800000u);
            // v in [2^-100, 2^100], t < 2^100, and r^2 zero or large enough for the residual
            odd |= bits - (27u << 23) > (200u << 23) || !(t < 1.2e30f) || (r2 < 1e-30f && r2 != 0.f);
        }
    }
    // after at most 64 gates (prod < 2^64); gh + gl = G ln 2 pi.  The terms meet
    // in the FP32 pair, each sum exact (an FP64 operation costs a warp 19 cycles
    // of the SM), ex ln2 as an exact product and its small rest (ln 2 as 355 / 512
    // and the rest, Cody & Waite 1980).
    __device__ __forceinline__ double ll(float gh, float gl) {
        plus(logf(prod));
        plus((float)ex * 0.693359375f);
        plus((float)ex * -2.12194440e-4f);
        plus(gh);
        const float hi = s + (e + gl);  // renormalised, so that the doubles' sum is exact
        const float lo = (s - hi) + (e + gl);
        return (double)(-0.5f * hi) + (double)(-0.5f * lo);
    }
};

// Converts the 16-byte core-matrix row of element chunk (r, kc) of the tile:
// chunk kc holds elements 16/ES * kc .. of row r.  src: that row's FP32
// values (nullptr: a padding row), zero past F.
template <int KIND>
__device__ __forceinline__ void stage_chunk(const float *__restrict__ src, int F, int kc, bool vec4,
                                            unsigned char *hi_row, unsigned char *lo_row) {
    using S = Split<KIND>;
    constexpr int KC = 16 / S::ES;  // elements per 16-byte core-matrix row
    float x[KC];
    const int k0 = kc * KC;
    if (src && vec4 && k0 + KC <= F) {
#pragma unroll
        for (int q = 0; q < KC; q += 4) {
            const float4 v = __ldg(reinterpret_cast<const float4 *>(src + k0 + q));
            x[q] = v.x;
            x[q + 1] = v.y;
            x[q + 2] = v.z;
            x[q + 3] = v.w;
        }
    } else {
#pragma unroll
        for (int q = 0; q < KC; ++q) x[q] = (src && k0 + q < F) ? __ldg(src + k0 + q) : 0.f;
    }
    typename S::T h[KC], l[KC];
#pragma unroll
    for (int q = 0; q < KC; ++q) S::run(x[q], h[q], l[q]);
    *reinterpret_cast<uint4 *>(hi_row) = *reinterpret_cast<const uint4 *>(h);
    *reinterpret_cast<uint4 *>(lo_row) = *reinterpret_cast<const uint4 *>(l);
}

// Register prefetch of a tile's spectra: thread tid owns chunks
// c = tid + j kThreads (j < JC = kTM NKC / kThreads), each chunk KC / 4 float4
// loads; a tile needs JC KC / 4 <= kPF of them per thread (F <= 64 for both
// splits) and F a multiple of 4 (16-byte rows).  The next tile's loads are
// issued before the current tile's epilogue, so their latency overlaps it.
// Chunk j is core-matrix row r7 + 8 q, column kc, with (q, kc) the quotient and
// remainder of (tid >> 3) + 32 j by NKC: the same for every tile, so each
// chunk's element offset and shared-memory offset are kept, not formed again
// (their arithmetic was a quarter of the kernel's instructions).
constexpr int kPF = 8;

template <int KIND>
struct TilePrefetch {
    static constexpr int KC = 16 / Split<KIND>::ES;  // elements per core-matrix row
    static constexpr int Q = KC / 4;                 // float4 loads per chunk
    static constexpr int JMAX = kPF / Q;             // chunks per thread
    float4 v[kPF];
    int at[JMAX];  // element offset in the tile << 8 of the chunk | its parts inside the row; negative: no chunk
    int to[JMAX];  // shared-memory offset

    __device__ __forceinline__ void init(int NKC, int F, uint32_t sbo, int tid) {
        const int jc = NKC * kTM / kThreads, r7 = tid & 7;
#pragma unroll
        for (int j = 0; j < JMAX; ++j) {
            const int i = (tid >> 3) + 32 * j, q = i / NKC, kc = i - q * NKC;
            const int parts = min(Q, max(0, (F - kc * KC + 3) / 4));
            at[j] = j < jc ? ((((r7 + 8 * q) * F + kc * KC) << 8) | parts) : -1;
            to[j] = q * (int)sbo + kc * 128 + r7 * 16;
        }
    }

    __device__ __forceinline__ void load(const float *__restrict__ imh, int P, int F, size_t row0) {
        const float *src = imh + row0 * F;
        const int end = P - (int)row0 >= kTM ? kTM * F : (P - (int)row0) * F;  // elements of this tile
#pragma unroll
        for (int j = 0; j < JMAX; ++j) {
            const int o = at[j] >> 8, parts = at[j] & 0xff;
#pragma unroll
            for (int p = 0; p < Q; ++p)
                v[j * Q + p] = at[j] >= 0 && o < end && p < parts
                                   ? __ldg(reinterpret_cast<const float4 *>(src + o + 4 * p))
                                   : make_float4(0.f, 0.f, 0.f, 0.f);
        }
    }

    __device__ __forceinline__ void store(unsigned char *hi, unsigned char *lo) const {
        using S = Split<KIND>;
        bool fin = true;
#pragma unroll
        for (int j = 0; j < kPF; ++j) {
            fin = fin && fabsf(v[j].x) < S::kFinite && fabsf(v[j].y) < S::kFinite && fabsf(v[j].z) < S::kFinite &&
                  fabsf(v[j].w) < S::kFinite;
        }
        if (fin)
            write<true>(hi, lo);
        else
            write<false>(hi, lo);
    }

    template <bool FINITE>
    __device__ __forceinline__ void write(unsigned char *hi, unsigned char *lo) const {
        using S = Split<KIND>;
#pragma unroll
        for (int j = 0; j < JMAX; ++j) {
            if (at[j] < 0) continue;
            float x[KC];
#pragma unroll
            for (int p = 0; p < Q; ++p) {
                x[4 * p] = v[j * Q + p].x;
                x[4 * p + 1] = v[j * Q + p].y;
                x[4 * p + 2] = v[j * Q + p].z;
                x[4 * p + 3] = v[j * Q + p].w;
            }
            typename S::T h[KC], l[KC];
#pragma unroll
            for (int p = 0; p < KC; ++p) {
                if constexpr (FINITE)
                    S::run_finite(x[p], h[p], l[p]);
                else
                    S::run(x[p], h[p], l[p]);
            }
            *reinterpret_cast<uint4 *>(hi + to[j]) = *reinterpret_cast<const uint4 *>(h);
            *reinterpret_cast<uint4 *>(lo + to[j]) = *reinterpret_cast<const uint4 *>(l);
        }
    }
};

// The same for rows that are not whole float4s (F not a multiple of 4): a
// tile's spectra are one contiguous block, thread tid takes its elements
// tid + 256 j, so the loads coalesce whatever F; element (row, column) advances
// by 256's quotient and remainder by F with one carry.  At most kFlat per
// thread (F <= 64).
constexpr int kFlat = 32;

template <int KIND>
struct FlatPrefetch {
    float v[kFlat];
    int F, n, row, col, dr, dc;

    __device__ __forceinline__ void init(int F_, int tid) {
        F = F_;
        n = kTM * F;
        row = tid / F;
        col = tid - row * F;
        dr = kThreads / F;
        dc = kThreads - dr * F;
    }

    __device__ __forceinline__ void load(const float *__restrict__ imh, int P, size_t row0) {
        const float *src = imh + row0 * F;
        const size_t left = ((size_t)P - row0) * F;
        const int m = left < (size_t)n ? (int)left : n;
#pragma unroll
        for (int j = 0; j < kFlat; ++j) {
            const int i = (int)threadIdx.x + j * kThreads;
            v[j] = i < m ? __ldg(src + i) : 0.f;
        }
    }

    __device__ __forceinline__ void store(uint32_t sbo, unsigned char *hi, unsigned char *lo) const {
        using S = Split<KIND>;
        constexpr int KC = 16 / S::ES;
        int r = row, c = col;
#pragma unroll
        for (int j = 0; j < kFlat; ++j) {
            if ((int)threadIdx.x + j * kThreads < n) {
                const uint32_t o = (uint32_t)(r >> 3) * sbo + (uint32_t)(c / KC) * 128u + (uint32_t)(r & 7) * 16u +
                                   (uint32_t)(c % KC) * S::ES;
                typename S::T h, l;
                S::run(v[j], h, l);
                *reinterpret_cast<typename S::T *>(hi + o) = h;
                *reinterpret_cast<typename S::T *>(lo + o) = l;
            }
            r += dr;
            c += dc;
            if (c >= F) {
                c -= F;
                ++r;
            }
        }
    }
};

// FLAT: the flat prefetch's registers (rows that are not whole float4s);
// otherwise the float4 one's, or none when the tile does not fit them.
// Software pipeline per CTA: once a tile's MMAs are done its operand buffer and
// the other accumulator are free, so the next tile is converted into shared
// memory and its MMAs issued, the spectra after it requested, and only then
// this tile's accumulator read: the tensor core and the loads run under the
// epilogue, one CTA barrier per tile.  2^20 spectra of 60 frequencies, TF32
// split, likelihood: 182 -> 113 us (a tile's chain of stage, fence, MMA, wait
// and epilogue took 14,600 cycles end to end; 8,700 warp instructions a tile
// are left at 56 % issue, 2.2 TB/s).
template <int KIND, bool FLAT>
__global__ void __launch_bounds__(kThreads, KIND == 0 || FLAT ? 2 : 3) gates_tc_kernel(TcArgs a) {
    using S = Split<KIND>;
    constexpr int ES = S::ES;
    constexpr int KI = 32 / ES;  // K of one MMA: two core matrices
    constexpr int KC = 16 / ES;  // elements per core-matrix row
    extern __shared__ unsigned char smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t pad = ((raw + 1023u) & ~1023u) - raw;
    unsigned char *base = smem_raw + pad;
    const int NKC = a.KP / KC;                // core-matrix columns (16-byte chunks per row)
    const uint32_t sbo = (uint32_t)NKC * 128u;  // same for A and B
    const uint32_t a_bytes = (uint32_t)kTM * a.KP * ES, b_bytes = (uint32_t)a.N * a.KP * ES;
    unsigned char *Ahi = base, *Alo = base + a_bytes, *Bhi = base + 2 * a_bytes, *Blo = Bhi + b_bytes;
    // [2][N]: the datum rows of this tile, (y high, y low, eps_an^2, 0); past G
    // (0, 0, 1, 0), which with the accumulator's zero there adds nothing
    float4 *ysplit = reinterpret_cast<float4 *>(Blo + b_bytes);
    float4 *llp = ysplit + 2 * AEM_MAX_GATES;  // [2][kTM]: the second column half's sums
    uint64_t *mbar_p = reinterpret_cast<uint64_t *>(llp + 2 * kTM);
    uint32_t *slot_p = reinterpret_cast<uint32_t *>(mbar_p + 1);
    int *abort_p = reinterpret_cast<int *>(slot_p + 1);
    const uint32_t mbar = smem_u32(mbar_p);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const bool vec4 = (a.F & 3) == 0 && ((reinterpret_cast<uintptr_t>(a.imh) & 15) == 0);

    if (tid == 0) {
        mbar_init(mbar, 1);
        *abort_p = 0;
    }
    __syncwarp();
    const uint32_t dcols = a.N <= 32 ? 32u : 64u;  // columns of one accumulator; two are allocated
    if (warp == 0) tmem_alloc(smem_u32(slot_p), 2 * dcols);
    // B = T (rows: gates, zero-padded to N; columns: frequencies, zero-padded to KP)
    for (int c = tid; c < a.N * NKC; c += kThreads) {
        const int r = (c & 7) + 8 * ((c >> 3) / NKC), kc = (c >> 3) % NKC;
        const uint32_t o = (uint32_t)(r >> 3) * sbo + (uint32_t)kc * 128u + (uint32_t)(r & 7) * 16u;
        stage_chunk<KIND>(r < a.G ? a.T + (size_t)r * a.F : nullptr, a.F, kc, false, Bhi + o, Blo + o);
    }
    if (FLAT) {  // columns past F stay zero
        for (uint32_t i = tid; i < 2 * a_bytes / 16; i += kThreads)
            reinterpret_cast<uint4 *>(base)[i] = make_uint4(0u, 0u, 0u, 0u);
    }
    tc_before_sync();
    __syncthreads();
    tc_after_sync();
    const uint32_t tbase = *slot_p;
    const uint32_t idesc = instr_desc(KIND == 0 ? 2u : 1u, (uint32_t)kTM, (uint32_t)a.N);
    const uint32_t ahi = smem_u32(Ahi), alo = smem_u32(Alo), bhi = smem_u32(Bhi), blo = smem_u32(Blo);
    const int ntiles = (a.P + kTM - 1) / kTM;
    const float em = (float)a.eps_mn;
    // P < 2^31 and obs_per >= 1: the datum row of model m is m / obs_per in 32-bit arithmetic
    const unsigned int obs_per = (unsigned int)a.obs_per;
    const unsigned int last_row = (unsigned int)(a.P - 1) / obs_per;
    const bool split_rows = a.y_obs && obs_per >= (unsigned int)kTM;

    typename std::conditional<FLAT, FlatPrefetch<KIND>, TilePrefetch<KIND>>::type pf;
    bool pf_ok = FLAT;
    if constexpr (FLAT) {
        pf.init(a.F, tid);
    } else {
        pf_ok = vec4 && NKC * kTM / kThreads * TilePrefetch<KIND>::Q <= kPF;
        if (pf_ok) pf.init(NKC, a.F, sbo, tid);
    }
    auto request = [&](int tile) {
        if (!pf_ok || tile >= ntiles) return;
        if constexpr (FLAT)
            pf.load(a.imh, a.P, (size_t)tile * kTM);
        else
            pf.load(a.imh, a.P, a.F, (size_t)tile * kTM);
    };
    // the tile's spectra as high / low operands (rows past P and columns past F
    // are zero); consecutive lanes fill consecutive 16-byte rows of one core matrix
    auto stage = [&](int tile) {
        if (pf_ok) {
            if constexpr (FLAT)
                pf.store(sbo, Ahi, Alo);
            else
                pf.store(Ahi, Alo);
        } else {
            for (int c = tid; c < kTM * NKC; c += kThreads) {
                const int r = (c & 7) + 8 * ((c >> 3) / NKC), kc = (c >> 3) % NKC;
                const size_t m = (size_t)tile * kTM + r;
                const uint32_t o = (uint32_t)(r >> 3) * sbo + (uint32_t)kc * 128u + (uint32_t)(r & 7) * 16u;
                stage_chunk<KIND>(m < (size_t)a.P ? a.imh + m * a.F : nullptr, a.F, kc, vec4, Ahi + o, Alo + o);
            }
        }
        fence_async_smem();
    };
    auto issue = [&](uint32_t acc) {
        for (int ks = 0; ks < a.KP / KI; ++ks) {
            const uint32_t off = (uint32_t)ks * 256u;
            const uint64_t dah = smem_desc(ahi + off, 128u, sbo), dal = smem_desc(alo + off, 128u, sbo);
            const uint64_t dbh = smem_desc(bhi + off, 128u, sbo), dbl = smem_desc(blo + off, 128u, sbo);
            mma<KIND>(acc, dah, dbh, idesc, ks > 0 ? 1u : 0u);
            mma<KIND>(acc, dah, dbl, idesc, 1u);
            mma<KIND>(acc, dal, dbh, idesc, 1u);
        }
        mma_commit(mbar);
    };

    const int quarter = warp & 3, half = warp >> 2, row = quarter * 32 + lane;
    uint32_t phase = 0;
    const int first_tile = (int)blockIdx.x, step = (int)gridDim.x;
    bool pending = !a.skip_mma;  // an MMA chain committed and not yet observed complete
    request(first_tile);
    stage(first_tile);
    tc_before_sync();
    __syncthreads();
    tc_after_sync();
    if (tid == 0 && pending) issue(tbase);
    request(first_tile + step);
    unsigned int have_row = 0xffffffffu;  // the datum row ysplit begins with
    LlAcc acc;          // of the tile before, until its other half's sums are there
    size_t acc_m = 0;
    bool acc_valid = false;
    // the two halves' sums meet in shared memory, added in a fixed order by the first half's thread
    auto finish = [&](int buf) {
        if (a.ll && half == 0 && acc_valid) {
            const float4 o = llp[buf * kTM + row];
            float s1, e1;
            two_sum(acc.s, o.x, s1, e1);
            acc.s = s1;
            acc.e = (acc.e + o.y) + e1;
            acc.prod *= o.z;
            acc.ex += __float_as_int(o.w);
            a.ll[acc_m] = acc.ll(a.gh, a.gl);
        }
    };
    int buf = 0;
    for (int tile = first_tile; tile < ntiles; tile += step, buf ^= 1) {
        const size_t row0 = (size_t)tile * kTM;
        const bool done = mbar_wait_bounded(mbar, phase, a.spins);
        if (!done) atomicExch(abort_p, 1);
        // the datum rows this tile's models use, as float pairs (at most two
        // when models_per_row >= the tile; otherwise the epilogue splits per model)
        const unsigned int s0 = last_row == 0 ? 0u : (unsigned int)row0 / obs_per;
        const bool new_row = split_rows && s0 != have_row;  // CTA-uniform
        const bool more = tile + step < ntiles;
        if (done && more) stage(tile + step);
        tc_before_sync();
        __syncthreads();
        tc_after_sync();
        finish(buf ^ 1);
        acc_valid = false;
        if (*abort_p) break;
        phase ^= 1u;
        pending = more;
        if (tid == 0 && more) issue(tbase + (uint32_t)(buf ^ 1) * dcols);
        request(tile + 2 * step);
        if (new_row) {  // the epilogue before has been left by every thread
            for (int i = tid; i < 2 * a.N; i += kThreads) {
                const int two = i >= a.N ? 1 : 0, g = i - two * a.N;
                const unsigned int srow = s0 + (unsigned int)two;
                float4 rec = make_float4(0.f, 0.f, 1.f, 0.f);
                if (g < a.G) {
                    const double y = a.y_obs[(size_t)(srow <= last_row ? srow : last_row) * a.G + g];
                    const float hi = (float)y;
                    rec = make_float4(hi, (float)(y - (double)hi), (float)(a.eps_an[g] * a.eps_an[g]), 0.f);
                }
                ysplit[i] = rec;
            }
            have_row = s0;
            __syncthreads();
        }
        // epilogue: this thread's model is row 32 (warp mod 4) + lane of the
        // tile; warps 0-3 take the first half of the gate columns, 4-7 the second
        const size_t m = row0 + (size_t)row;
        const bool valid = m < (size_t)a.P;
        // with split rows the tile spans datum rows s0 and s0 + 1 at most
        const unsigned int srow =
            !valid ? 0u
                   : split_rows ? s0 + ((unsigned int)m >= (s0 + 1u) * obs_per ? 1u : 0u) : (unsigned int)m / obs_per;
        const float4 *yrow = ysplit + (split_rows ? (srow - s0) * (unsigned int)a.N : 0u);
        const double *yd = (a.y_obs && !split_rows) ? a.y_obs + (size_t)srow * a.G : nullptr;
        const int c_lo = half * (a.N / 2), c_hi = c_lo + a.N / 2;
        auto columns = [&](auto exact) {
            constexpr bool EXACT = decltype(exact)::value;
            acc = LlAcc();
            for (int c = c_lo; c < c_hi; c += 8) {
                float v[8];
                tmem_ld8(tbase + (uint32_t)buf * dcols + ((uint32_t)(quarter * 32) << 16) + (uint32_t)c, v);
                if (!EXACT && a.gates && valid) {
#pragma unroll
                    for (int q = 0; q < 8; ++q)
                        if (c + q < a.G) a.gates[m * a.G + c + q] = v[q];
                }
                if (split_rows) {  // columns past G and rows past P are harmless
#pragma unroll
                    for (int q = 0; q < 8; ++q) {
                        const float4 y = yrow[c + q];
                        if (!EXACT || c + q < a.G) acc.add<EXACT>(v[q], make_float2(y.x, y.y), y.z, em);
                    }
                } else if (yd && valid) {
                    for (int q = 0; q < 8 && c + q < a.G; ++q) {
                        const double yv = yd[c + q];
                        const float hi = (float)yv, ea = (float)(a.eps_an[c + q] * a.eps_an[c + q]);
                        acc.add<EXACT>(v[q], make_float2(hi, (float)(yv - (double)hi)), ea, em);
                    }
                }
            }
        };
        columns(std::false_type{});
        if (__any_sync(0xffffffffu, acc.odd)) columns(std::true_type{});
        acc_m = m;
        acc_valid = valid;
        if (a.ll && half == 1) llp[buf * kTM + row] = make_float4(acc.s, acc.e, acc.prod, __int_as_float(acc.ex));
    }
    tc_before_sync();
    __syncthreads();
    tc_after_sync();
    if (*abort_p) {
        if (tid == 0) atomicExch(a.status, (int)AEM_ERR_TIMEOUT);
        if (pending) mbar_wait_bounded(mbar, phase);  // our own MMAs, once more with the full limit
    } else {
        finish(buf ^ 1);
    }
    tc_before_sync();
    __syncthreads();
    tc_after_sync();
    if (warp == 0) tmem_dealloc(tbase, 2 * dcols);
}

// FP32 CUDA-core form of the same transform (for comparison): one thread per
// model, T staged in shared memory, the same FP32 likelihood terms.
__global__ void gates_fp32_kernel(TcArgs a) {
    extern __shared__ float Ts[];
    __shared__ float ea2[AEM_MAX_GATES];
    for (int i = threadIdx.x; i < a.G * a.F; i += blockDim.x) Ts[i] = a.T[i];
    if (a.eps_an)
        for (int g = threadIdx.x; g < a.G; g += blockDim.x) ea2[g] = (float)(a.eps_an[g] * a.eps_an[g]);
    __syncthreads();
    const float em = (float)a.eps_mn;
    for (size_t m = (size_t)blockIdx.x * blockDim.x + threadIdx.x; m < (size_t)a.P; m += (size_t)gridDim.x * blockDim.x) {
        const float *x = a.imh + m * a.F;
        const double *y = a.y_obs ? a.y_obs + (m / (size_t)a.obs_per) * a.G : nullptr;
        LlAcc acc;
        for (int g = 0; g < a.G; ++g) {
            float s = 0.f;
            for (int k = 0; k < a.F; ++k) s = fmaf(Ts[g * a.F + k], x[k], s);
            if (a.gates) a.gates[m * a.G + g] = s;
            if (y) {
                const float hi = (float)y[g];
                acc.add<true>(s, make_float2(hi, (float)(y[g] - (double)hi)), ea2[g], em);
            }
        }
        if (a.ll) a.ll[m] = acc.ll(a.gh, a.gl);
    }
}

inline int round_up(int x, int m) { return (x + m - 1) / m * m; }

// CTAs per SM of the tensor-core transform.  The occupancy query has reported
// one CTA per SM for the TF32 tile where two fit (the profiler's shared-memory
// limit says two); take the count the SM's shared memory, registers and tensor
// memory allow when it is larger.
template <class Kernel>
int tc_resident(const aem_system *sys, int mode, Kernel kern, size_t smem, int ncols, int *out) {
    int per_sm = sys->tc_ctas[mode].load(std::memory_order_relaxed);
    if (per_sm == 0) {
        std::atomic<int> asked{0};
        if (const int rc = resident_ctas(&asked, kern, kThreads, smem, sys->device, &per_sm)) return rc;
        if (per_sm > 0) {
            int smem_sm = 0, reserved = 0;
            AEM_CUDA_TRY(cudaDeviceGetAttribute(&smem_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, sys->device));
            AEM_CUDA_TRY(cudaDeviceGetAttribute(&reserved, cudaDevAttrReservedSharedMemoryPerBlock, sys->device));
            cudaFuncAttributes fa{};
            AEM_CUDA_TRY(cudaFuncGetAttributes(&fa, kern));
            int by_smem = smem_sm / (int)(smem + (size_t)reserved);
            const int by_regs = fa.numRegs > 0 ? 65536 / (fa.numRegs * kThreads) : 1;
            const int by_tmem = 512 / ncols;
            if (by_smem > by_regs) by_smem = by_regs;
            if (by_smem > by_tmem) by_smem = by_tmem;
            if (by_smem > per_sm) per_sm = by_smem;
            sys->tc_ctas[mode].store(per_sm, std::memory_order_relaxed);
        }
    }
    *out = per_sm;
    return AEM_OK;
}

}  // namespace

int gates_from_spectrum(const aem_system *sys, const float *imh, int P, int mode, const double *y_obs,
                        int obs_per, const double *eps_an, double eps_mn, float *gates, double *ll,
                        cudaStream_t stream) {
    const SystemTables &h = sys->host;
    const double gconst = h.G * kLn2Pi;
    TcArgs a{imh, P, h.F, h.G, 0, 0, 0, sys->d_T_f, y_obs, obs_per > 0 ? obs_per : 1, eps_an, eps_mn, gates, ll,
             sys->d_status, (float)gconst, (float)(gconst - (double)(float)gconst), sys->wait_spins ? sys->wait_spins : kSpinLimit, sys->wait_skip_mma};
    if (mode == AEM_GATES_FP32) {
        const size_t smem = sizeof(float) * (size_t)h.G * h.F;
        int grid = (int)((P + 255) / 256);
        if (grid > sys->num_sms * 8) grid = sys->num_sms * 8;
        gates_fp32_kernel<<<grid, 256, smem, stream>>>(a);
        AEM_CUDA_TRY(cudaGetLastError());
        return AEM_OK;
    }
    const bool tf32 = mode == AEM_GATES_TF32_SPLIT;
    const int ES = tf32 ? 4 : 2, KI = 32 / ES;
    a.KP = round_up(h.F, KI);
    a.N = round_up(h.G, 16);
    a.ncols = 2 * (a.N <= 32 ? 32 : 64);
    const size_t smem = (size_t)2 * (kTM + a.N) * a.KP * ES + 1024 + sizeof(float4) * 2 * AEM_MAX_GATES +
                        sizeof(float4) * 2 * kTM + 64;
    // rows of whole float4s take the float4 prefetch, others (up to 64
    // frequencies, kFlat registers) the flat one
    const bool flat = (h.F & 3) != 0 && h.F <= 2 * kFlat;
    auto kern = tf32 ? (flat ? gates_tc_kernel<0, true> : gates_tc_kernel<0, false>)
                     : (flat ? gates_tc_kernel<1, true> : gates_tc_kernel<1, false>);
    int per_sm = 0;
    if (const int rc = tc_resident(sys, mode, kern, smem, a.ncols, &per_sm)) return rc;
    if (per_sm < 1) return fail(AEM_ERR_UNSUPPORTED, "aem_gates_from_spectrum: tile does not fit in shared memory");
    const int ntiles = (P + kTM - 1) / kTM;
    int grid = sys->num_sms * per_sm;
    if (grid > ntiles) grid = ntiles;
    kern<<<grid, kThreads, smem, stream>>>(a);
    AEM_CUDA_TRY(cudaGetLastError());
    return AEM_OK;
}

}  // namespace aem

using namespace aem;

extern "C" int aem_gates_from_spectrum(const aem_system *sys, const float *imh, int n_models, int mode,
                                       const double *y_obs, const double *eps_an, double eps_mn, float *gates,
                                       double *ll, void *stream) {
    if (!sys) return fail(AEM_ERR_INVALID_ARG, "aem_gates_from_spectrum: sys is NULL");
    if (n_models < 0) return fail(AEM_ERR_INVALID_ARG, "aem_gates_from_spectrum: n_models < 0");
    if (mode != AEM_GATES_FP32 && mode != AEM_GATES_TF32_SPLIT && mode != AEM_GATES_BF16_SPLIT)
        return fail(AEM_ERR_INVALID_ARG, "aem_gates_from_spectrum: unknown mode");
    if (n_models == 0) return AEM_OK;
    if (!imh || (!gates && !ll) || (ll && (!y_obs || !eps_an)))
        return fail(AEM_ERR_INVALID_ARG, "aem_gates_from_spectrum: NULL pointer");
    return gates_from_spectrum(sys, imh, n_models, mode, y_obs, n_models, eps_an, eps_mn, gates, ll,
                               (cudaStream_t)stream);
}

extern "C" int aem_loglik_f32_tc(const aem_system *sys, const aem_models_f32 *models, const double *y_obs,
                                 const double *eps_an, double eps_mn, int mode, float *imh_work, double *ll,
                                 float *gates, void *stream) {
    if (!sys || !models) return fail(AEM_ERR_INVALID_ARG, "aem_loglik_f32_tc: NULL system or models");
    if (models->n_models == 0) return AEM_OK;
    if (!imh_work || !ll || !y_obs || !eps_an) return fail(AEM_ERR_INVALID_ARG, "aem_loglik_f32_tc: NULL pointer");
    int rc = aem_forward_f32(sys, models, nullptr, imh_work, stream);
    if (rc) return rc;
    return aem_gates_from_spectrum(sys, imh_work, models->n_models, mode, y_obs, eps_an, eps_mn, gates, ll, stream);
}

extern "C" int aem_debug_bounded_wait(aem_system *sys, unsigned int spins, int skip_first_mma) {
    if (!sys || (skip_first_mma != 0 && skip_first_mma != 1))
        return fail(AEM_ERR_INVALID_ARG, "aem_debug_bounded_wait: NULL system or skip_first_mma not 0 / 1");
    sys->wait_spins = spins;
    sys->wait_skip_mma = skip_first_mma;
    return AEM_OK;
}

extern "C" int aem_system_status(const aem_system *sys, int *status) {
    if (!sys || !status) return fail(AEM_ERR_INVALID_ARG, "aem_system_status: NULL argument");
    int v = 0;
    AEM_CUDA_TRY(cudaMemcpy(&v, sys->d_status, sizeof(int), cudaMemcpyDeviceToHost));
    if (v != 0) AEM_CUDA_TRY(cudaMemset(sys->d_status, 0, sizeof(int)));
    *status = v;
    return AEM_OK;
}
