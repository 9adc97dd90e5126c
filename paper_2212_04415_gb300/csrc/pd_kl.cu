// pd_kl.cu -- truncated-KL field sampling on the tensor cores (Section 3):
// g[b][i] = sum_k Psi[i][k] xi[b][k], Psi = Phi diag(sqrt(lambda)), followed by
// the marginal transform (lognormal, or the Weibull copula of Section 6),
// written as FP32 node fields [B][N].
//
// The contraction runs as tcgen05.mma kind::tf32 with FP32 accumulators in
// tensor memory. TF32 keeps 11 significant bits, so each operand is split
// into hi = tf32(x) and lo = tf32(x - hi) and the product is taken as
// hi*hi + hi*lo + lo*hi (three MMAs; the dropped lo*lo term is below
// 2^-22 relative), which gives FP32-class accuracy.
//
// One persistent CTA an SM keeps the split coefficients of its sample tile (up
// to 256 samples) in shared memory and walks over tiles of 128 nodes (the MMA's
// M), one warp role per stage:
//   producer    Psi chunks of 32 modes (one 128-byte swizzle atom of FP32) by
//               TMA, up to six stages deep
//   converters  the chunk split into TF32 hi (in place) and lo, elementwise, so
//               the swizzle does not matter; Psi is read from memory once, in FP32
//   issuer      4 x 3 MMAs per chunk into one of two accumulators in tensor memory
//   epilogue    first the coefficients, narrowed and split from FP64; then
//               tcgen05.ld, the marginal transform, stores coalesced along nodes
// so copies, splitting, products and stores of successive tiles overlap. The
// sum over modes runs in one order whatever the tile shape, so a sample's field
// does not depend on the batch.
// Bound by the field writes with the lognormal marginal (24 epilogue warps for
// the latency of tcgen05.ld and the stores), by instruction issue with Weibull's
// erfcf, logf and powf (24 instead of 16 epilogue warps, taking 16-column units
// in turn across tiles: 355 to 315 us). With 64 modes on GB300, L2 dirty before
// each call, against stages in turn, three CTAs an SM and Psi stored as hi and lo:
//   224,000 nodes x 256 samples        74 us (100);  Weibull 315 (325)
//   224,000 x 100                      53    (66)
//   28,000 x 1                         20    (23)
//   28,000 x 256                       29    (31)
// (286 MB of Psi and fields take 42 us at the copy rate. A call for 28,000 x 1, with
// the drawing of its coefficients and the host's part, shows no gain: 30 to 38 us
// against 32 to 36, runs of either differing by 7 to 14 %.)
// Every wait on an mbarrier has an iteration limit; on expiry the CTA records
// an error, writes NaN into its remaining tiles and still waits (bounded) for
// its own copies and MMAs before it frees tensor memory.
#include <cuda.h>

#include <algorithm>
#include <climits>
#include <mutex>

#include "pd_internal.cuh"

namespace pdi {

constexpr int kKlM = 128;          // nodes per tile (MMA M)
constexpr int kKlChunk = 32;       // modes per chunk (128 B of FP32)
constexpr int kKlStages = 6;       // Psi chunks in flight, at most
constexpr int kKlConv = 4;         // converter warps (2 .. 5)
constexpr int kKlEpi = 24;         // epilogue warps (6 .. 29): six for each quarter of the tensor memory lanes
constexpr int kKlThreads = 32 * (2 + kKlConv + kKlEpi);
constexpr size_t kKlSmem = 226 * 1024;  // dynamic shared memory, at most
constexpr uint32_t kSpinLimit = 1u << 22;

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ float tf32_rna(float x) {
    uint32_t r;
    asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
    return __uint_as_float(r);
}

__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint64_t *bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint64_t *bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

// Bounded wait for the phase with the given parity; false when the limit
// expired or another thread of the CTA has given up (fail, or nullptr).
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, uint32_t parity, const volatile int *fail) {
    const uint32_t a = smem_u32(bar);
    for (uint32_t it = 0; it < kSpinLimit; ++it) {
        uint32_t ok;
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(ok)
            : "r"(a), "r"(parity)
            : "memory");
        if (ok) return true;
        if (fail && *fail) return false;
    }
    return false;
}

__device__ __forceinline__ void tma_load_2d(void *dst, const CUtensorMap *tm, int x, int y, uint64_t *bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::
            "r"(smem_u32(dst)),
        "l"((uint64_t)tm), "r"(x), "r"(y), "r"(smem_u32(bar))
        : "memory");
}

// Shared-memory matrix descriptor of a K-major operand in the 128-byte
// swizzle: rows of 128 B, 8-row groups 1024 B apart (stride byte offset),
// descriptor version 1, swizzle mode 2 (128B).
__device__ __forceinline__ uint64_t sw128_desc(uint32_t saddr) {
    uint64_t d = 0;
    d |= (uint64_t)((saddr & 0x3FFFF) >> 4);
    d |= (uint64_t)1 << 16;            // leading byte offset (unused for swizzled K-major)
    d |= (uint64_t)(1024 >> 4) << 32;  // stride byte offset
    d |= (uint64_t)1 << 46;            // descriptor version
    d |= (uint64_t)2 << 61;            // 128B swizzle
    return d;
}

// Instruction descriptor, kind::tf32: FP32 accumulator, TF32 A and B, both
// K-major, N = n, M = 128.
__host__ __device__ constexpr uint32_t tf32_idesc(int n) {
    return (1u << 4) | (2u << 7) | (2u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(kKlM >> 4) << 24);
}

__device__ __forceinline__ void mma_tf32(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                         uint32_t accumulate) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem_d),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
}

__device__ __forceinline__ void mma_commit(uint64_t *bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
                 : "memory");
}

__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float v[16]) {
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
        "%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int q = 0; q < 16; ++q) v[q] = __uint_as_float(r[q]);
}

// Psi padded to rows of Kp modes (only when the rows of K are no multiple of
// 16 bytes, as TMA needs, or shorter than a chunk).
__global__ void k_pad_psi(long long N, int K, int Kp, const float *phi, float *out) {
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= N * Kp) return;
    const long long i = t / Kp;
    const int k = (int)(t % Kp);
    out[t] = k < K ? phi[i * K + k] : 0.0f;
}

// FP64 to FP32, round to nearest even, with integer operations: conversions
// run on the FP64 pipe (2 lanes an SM on this part). Results in the normal
// range only; the rest takes the conversion.
__device__ __forceinline__ float narrow(double x) {
    const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x), e = (hi >> 20) & 0x7ffu;
    if (e < 897u || e > 1149u) return (float)x;
    const uint32_t m = ((e - 896u) << 23) | ((hi & 0xfffffu) << 3) | (lo >> 29), rest = lo & 0x1fffffffu;
    const uint32_t up = (rest > 0x10000000u || (rest == 0x10000000u && (m & 1u))) ? 1u : 0u;
    return __uint_as_float((hi & 0x80000000u) | (m + up));
}

struct KlArgs {
    long long N, N2;    // nodes of the level and of the coarse level (0: none)
    int K, Kp, B, nt;
    int nbt;            // sample tiles
    int stages;         // Psi chunks in flight
    long long n_first, n_tiles;  // node tiles of the level, and with the coarse level's after them
    int marginal;
    float mu, sig, wscale, winvm;
    const double *xi;   // [B][K]
    float *out, *out2;  // [B][N], [B][N2]
    int *err;
};

__global__ void __launch_bounds__(kKlThreads, 1) k_sample_tc(const __grid_constant__ CUtensorMap tm_psi,
                                                                 const __grid_constant__ CUtensorMap tm_psi2,
                                                                 const KlArgs a) {
    extern __shared__ __align__(1024) uint8_t kl_smem_raw[];
    __shared__ uint64_t bar_raw[kKlStages], bar_split[kKlStages], bar_free[kKlStages];  // chunk arrived, split, consumed
    __shared__ uint64_t bar_acc[2], bar_out[2];                                          // accumulator ready, drained
    __shared__ uint64_t bar_coef, bar_drain;                                             // coefficients split, all MMAs done
    __shared__ uint32_t s_tmem;
    __shared__ volatile int s_fail;
    uint8_t *sm = (uint8_t *)(((uintptr_t)kl_smem_raw + 1023) & ~(uintptr_t)1023);
    // stages: hi (as copied, then split in place) and lo, 128 rows x 128 B each
    const auto stage_hi = [&](int s) { return sm + (size_t)s * 2 * kKlM * 128; };
    const auto stage_lo = [&](int s) { return stage_hi(s) + kKlM * 128; };
    uint8_t *sB_hi = sm + (size_t)a.stages * 2 * kKlM * 128;  // [chunk] nt rows x 128 B
    const int nchunks = a.Kp / kKlChunk;
    uint8_t *sB_lo = sB_hi + (size_t)nchunks * a.nt * 128;

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int b0 = (int)(blockIdx.x % (unsigned)a.nbt) * a.nt;
    const long long t0 = blockIdx.x / (unsigned)a.nbt, tstep = gridDim.x / (unsigned)a.nbt;  // node tiles of this CTA
    const int acols = a.nt < 32 ? 32 : a.nt;  // columns of an accumulator: a power of two by construction (host)

    if (tid == 0) {
        for (int s = 0; s < kKlStages; ++s) {
            mbar_init(&bar_raw[s], 1);
            mbar_init(&bar_split[s], 32 * kKlConv);
            mbar_init(&bar_free[s], 1);
        }
        for (int q = 0; q < 2; ++q) {
            mbar_init(&bar_acc[q], 1);
            mbar_init(&bar_out[q], kKlEpi);
        }
        mbar_init(&bar_coef, kKlEpi);
        mbar_init(&bar_drain, 1);
        s_fail = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem)),
                     "r"(2 * acols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = s_tmem;
    uint32_t issued = 0;   // chunks (producer) or committed batches (issuer) of this role
    // chunk n of the CTA uses stage n % stages, phase n / stages
    if (warp == 0) {
        if (lane == 0) {
            for (long long t = t0; t < a.n_tiles && !s_fail; t += tstep) {
                for (int c = 0; c < nchunks; ++c) {
                    const int s = issued % a.stages;
                    const uint32_t ph = issued / a.stages;
                    if (ph > 0 && !mbar_wait(&bar_free[s], (ph - 1) & 1u, &s_fail)) {
                        s_fail = 1;
                        break;
                    }
                    mbar_expect_tx(&bar_raw[s], kKlM * 128u);
                    if (t < a.n_first)
                        tma_load_2d(stage_hi(s), &tm_psi, c * kKlChunk, (int)(t * kKlM), &bar_raw[s]);
                    else
                        tma_load_2d(stage_hi(s), &tm_psi2, c * kKlChunk, (int)((t - a.n_first) * kKlM), &bar_raw[s]);
                    ++issued;
                }
            }
        }
    } else if (warp == 1) {
        if (lane == 0) {
            const uint32_t idesc = tf32_idesc(a.nt);
            uint32_t n = 0;
            bool ok = mbar_wait(&bar_coef, 0u, &s_fail);
            for (long long t = t0; t < a.n_tiles && ok; t += tstep) {
                const int q = issued & 1;
                const uint32_t ph = issued >> 1;
                if (ph > 0 && !mbar_wait(&bar_out[q], (ph - 1) & 1u, &s_fail)) break;
                const uint32_t acc = tmem + (uint32_t)(q * acols);
                for (int c = 0; c < nchunks; ++c, ++n) {
                    const int s = n % a.stages;
                    if (!mbar_wait(&bar_split[s], (n / a.stages) & 1u, &s_fail)) {
                        ok = false;
                        break;
                    }
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    const uint32_t aH = smem_u32(stage_hi(s)), aL = smem_u32(stage_lo(s));
                    const uint32_t bH = smem_u32(sB_hi + (size_t)c * a.nt * 128), bL = smem_u32(sB_lo + (size_t)c * a.nt * 128);
#pragma unroll
                    for (int k = 0; k < kKlChunk / 8; ++k) {  // K = 8 per MMA: 32 B along the row
                        const uint32_t o = 32u * k;
                        const uint32_t acc0 = (c > 0 || k > 0) ? 1u : 0u;
                        mma_tf32(acc, sw128_desc(aL + o), sw128_desc(bH + o), idesc, acc0);
                        mma_tf32(acc, sw128_desc(aH + o), sw128_desc(bL + o), idesc, 1u);
                        mma_tf32(acc, sw128_desc(aH + o), sw128_desc(bH + o), idesc, 1u);
                    }
                    mma_commit(&bar_free[s]);
                }
                if (ok) mma_commit(&bar_acc[q]);
                ++issued;
            }
            if (issued != (uint32_t)((a.n_tiles - t0 + tstep - 1) / tstep) || !ok) s_fail = 2;
            mma_commit(&bar_drain);  // all MMAs of the CTA
        }
    } else if (warp < 2 + kKlConv) {
        const int ct = tid - 64;
        uint32_t n = 0;
        bool ok = true;
        for (long long t = t0; t < a.n_tiles && ok; t += tstep) {
            for (int c = 0; c < nchunks; ++c, ++n) {
                const int s = n % a.stages;
                if (!mbar_wait(&bar_raw[s], (n / a.stages) & 1u, &s_fail)) {
                    s_fail = 1;
                    ok = false;
                    break;
                }
                float4 *hi = (float4 *)stage_hi(s), *lo = (float4 *)stage_lo(s);
#pragma unroll
                for (int q = 0; q < kKlM * 128 / 16 / (32 * kKlConv); ++q) {
                    const int e = ct + q * 32 * kKlConv;
                    const float4 x = hi[e];
                    const float4 h = make_float4(tf32_rna(x.x), tf32_rna(x.y), tf32_rna(x.z), tf32_rna(x.w));
                    hi[e] = h;
                    lo[e] = make_float4(tf32_rna(x.x - h.x), tf32_rna(x.y - h.y), tf32_rna(x.z - h.z), tf32_rna(x.w - h.w));
                }
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                mbar_arrive(&bar_split[s]);
            }
        }
    } else {
        const int quarter = warp & 3;                      // tensor memory lanes 32 quarter .. + 31
        // the coefficients of the sample tile: split, K-major, 128-byte swizzle
        // (16-byte units of a row xor the row's position in its group of 8)
        for (int b = warp - 2 - kKlConv; b < a.nt; b += kKlEpi) {
            const size_t at = (size_t)b * 128 + (((lane >> 2) ^ (b & 7)) << 4) + (lane & 3) * 4;
            for (int c = 0; c < nchunks; ++c) {
                const int k = c * kKlChunk + lane;
                const float x = b0 + b < a.B && k < a.K ? narrow(a.xi[(size_t)(b0 + b) * a.K + k]) : 0.0f;
                const float h = tf32_rna(x);
                *(float *)(sB_hi + (size_t)c * a.nt * 128 + at) = h;
                *(float *)(sB_lo + (size_t)c * a.nt * 128 + at) = tf32_rna(x - h);
            }
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncwarp();
        if (lane == 0) mbar_arrive(&bar_coef);
        // groups of four warps take the accumulators' 16-column units in turn, across tiles
        constexpr int kG = kKlEpi / 4;
        const int units = a.nt / 16;
        int u = (warp - 2 - kKlConv) / 4;  // next unit of this group, counted from the current tile's first
        uint32_t n = 0;
        for (long long t = t0; t < a.n_tiles; t += tstep, ++n, u -= units) {
            const int q = n & 1;
            const bool first = t < a.n_first;
            const long long N = first ? a.N : a.N2, i = (first ? t : t - a.n_first) * kKlM + quarter * 32 + lane;
            float *const out = first ? a.out : a.out2;
            const bool ok = __all_sync(0xffffffffu, mbar_wait(&bar_acc[q], (n >> 1) & 1u, &s_fail));
            if (!ok) {
                s_fail = 2;
                for (; u < units; u += kG)
                    for (int b = b0 + 16 * u; i < N && b < min(a.B, b0 + 16 * u + 16); ++b)
                        out[(size_t)b * N + i] = __int_as_float(0x7fc00000);
                continue;
            }
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint32_t base = tmem + (uint32_t)(q * acols) + ((uint32_t)(quarter * 32) << 16);
            if (u >= units && lane == 0) mbar_arrive(&bar_out[q]);  // none of this tile's
            for (; u < units; u += kG) {
                const int j0 = 16 * u;
                float v[16];
                tmem_ld16(base + (uint32_t)j0, v);
                if (u + kG >= units) {  // the warp's part is in registers
                    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&bar_out[q]);
                }
                float *o = out + (size_t)(b0 + j0) * N + i;
                const int nb = i < N ? min(16, a.B - b0 - j0) : 0;  // samples of this lane's node to write
                if (a.marginal == PD_MARG_LOGNORMAL) {
#pragma unroll
                    for (int w = 0; w < 16; ++w) v[w] = expf(a.mu + a.sig * v[w]);
                } else {
#pragma unroll
                    for (int w = 0; w < 16; ++w) {
                        const float q1 = 0.5f * erfcf(v[w] * 0.70710678118654752f);  // 1 - Phi(g)
                        v[w] = a.wscale * powf(-logf(q1), a.winvm);
                    }
                }
                if (nb == 16) {
#pragma unroll
                    for (int w = 0; w < 16; ++w, o += N) __stcs(o, v[w]);
                } else {
#pragma unroll
                    for (int w = 0; w < 16; ++w, o += N)
                        if (w < nb) __stcs(o, v[w]);
                }
            }
        }
    }
    // the CTA's own copies and MMAs end (bounded) before its memory is released
    if (warp == 0 && lane == 0 && s_fail) {
        for (uint32_t k = issued > (uint32_t)a.stages ? issued - a.stages : 0; k < issued; ++k)
            mbar_wait(&bar_raw[k % a.stages], (k / a.stages) & 1u, nullptr);
    }
    if (warp == 1 && lane == 0) mbar_wait(&bar_drain, 0u, nullptr);
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (tid == 0 && s_fail) atomicOr(a.err, s_fail);
    if (warp == 0) {
        __syncwarp();
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(2 * acols) : "memory");
    }
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static EncodeTiledFn encode_fn() {
    static std::once_flag once;
    static EncodeTiledFn fn = nullptr;
    std::call_once(once, [] {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = (EncodeTiledFn)p;
    });
    return fn;
}

// Rows of K modes (pitch floats apart) of FP32, K-major, read in boxes of 32
// modes x 128 rows, 128B swizzle; modes beyond K read as zero.
static int encode_psi(CUtensorMap *tm, const float *base, long long rows, int K, int pitch) {
    EncodeTiledFn enc = encode_fn();
    PD_REQUIRE(enc != nullptr, "cuTensorMapEncodeTiled is unavailable");
    const cuuint64_t dims[2] = {(cuuint64_t)K, (cuuint64_t)rows};
    const cuuint64_t strides[1] = {(cuuint64_t)pitch * sizeof(float)};
    const cuuint32_t box[2] = {(cuuint32_t)kKlChunk, (cuuint32_t)kKlM};
    const cuuint32_t estr[2] = {1, 1};
    const CUresult r = enc(tm, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, (void *)base, dims, strides, box, estr,
                           CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                           CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    PD_REQUIRE(r == CUDA_SUCCESS, "cuTensorMapEncodeTiled failed (%d)", (int)r);
    return PD_OK;
}

// Shared memory of a CTA: the stages, and hi and lo of nt samples x Kp modes.
static size_t kl_smem_bytes(int nt, int Kp, int stages) {
    return 1024 + (size_t)stages * 2 * kKlM * 128 + 2 * (size_t)nt * Kp * sizeof(float);
}

}  // namespace pdi

using namespace pdi;

struct KlOperand {
    CUtensorMap tm;          // 64-byte aligned by type
    float *psi = nullptr;    // padded copy of the basis, or nullptr (the caller's rows)
    int *err = nullptr;
    long long N = 0;
    int K = 0, Kp = 0;
    int sms = 0;
};

// phi: device [N][K], kept by the caller for the operand's lifetime.
int kl_operand_create(const float *phi, long long N, int K, KlOperand **out) {
    PD_REQUIRE(N >= 1 && K >= 1 && K <= 256, "1 <= K <= 256 and N >= 1 required");
    PD_REQUIRE(N < (1LL << 31), "N too large for the TMA coordinate");
    KlOperand *op = new KlOperand();
    op->N = N;
    op->K = K;
    op->Kp = (K + kKlChunk - 1) / kKlChunk * kKlChunk;
    int dev = 0;
    int rc = dalloc(&op->err, 1);
    if (rc == PD_OK && (cudaMemset(op->err, 0, sizeof(int)) != cudaSuccess || cudaGetDevice(&dev) != cudaSuccess ||
                        cudaDeviceGetAttribute(&op->sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess))
        rc = PD_ERR_CUDA;
    if (rc == PD_OK && (K % 4 != 0 || K < kKlChunk)) {
        rc = dalloc(&op->psi, (size_t)N * op->Kp);
        if (rc == PD_OK) {
            const long long n = N * op->Kp;
            k_pad_psi<<<(unsigned)((n + 255) / 256), 256>>>(N, K, op->Kp, phi, op->psi);
            if (cudaGetLastError() != cudaSuccess) rc = PD_ERR_CUDA;
        }
    }
    if (rc == PD_OK) rc = op->psi ? encode_psi(&op->tm, op->psi, N, op->Kp, op->Kp) : encode_psi(&op->tm, phi, N, K, K);
    if (rc == PD_OK) {
        static std::once_flag attr;
        std::call_once(attr, [] {
            cudaFuncSetAttribute(k_sample_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kKlSmem);
        });
        if (cudaGetLastError() != cudaSuccess) rc = PD_ERR_CUDA;
    }
    if (rc != PD_OK) {
        kl_operand_destroy(op);
        return rc;
    }
    *out = op;
    return PD_OK;
}

void kl_operand_destroy(KlOperand *op) {
    if (!op) return;
    cudaFree(op->psi);
    cudaFree(op->err);
    delete op;
}

int kl_operand_error(const KlOperand *op) {
    int h = 0;
    if (op && cudaMemcpy(&h, op->err, sizeof(int), cudaMemcpyDeviceToHost) != cudaSuccess) return -1;
    return h;
}

// Samples per tile: a power of two of at least 32 columns of tensor memory, at
// most 256 (two accumulators fill it), whose split coefficients take at most
// 128 KB (256 samples up to 64 modes, 128 up to 128, 64 up to 256). A CTA's time
// goes with its rounds, and a round's with its columns (transform and stores)
// plus the splitting and products of its chunks, about 32 columns' worth a chunk
// (measured; 16 and 64 choose the same or slower). So 224,000 nodes x 256
// samples take 256 columns, each node tile split once (74 us; 92 in tiles of
// 128), and 28,000 x 256, two rounds of 256 with the second half empty, three of
// 128 (30 us; 35).
static int pick_nt(long long n_tiles, int B, int Kp, int sms) {
    int best = 32;
    long long cost = LLONG_MAX;
    for (int nt = 32; nt <= 256 && nt * Kp <= 16384 && nt < 2 * B + 32; nt *= 2) {
        const long long nbt = (B + nt - 1) / nt, per = std::max<long long>(1, std::min<long long>(n_tiles, sms / nbt));
        const long long rounds = (n_tiles + per - 1) / per, waves = (per * nbt + sms - 1) / sms;
        const long long c = rounds * waves * (nt + Kp);
        if (c <= cost) {
            cost = c;
            best = nt;
        }
    }
    return best;
}

// op2, out2: the coarse level of the same field (same modes), or nullptr. Its
// tiles follow in the same launch: 224,000 nodes x 256 samples with the 28,000
// of the coarse level 77 us as one launch, 92 as two.
int kl_sample_tc(KlOperand *op, KlOperand *op2, const double *xi, int B, int marginal, double mu, double sig,
                 double wscale, double winvm, float *out, float *out2, cudaStream_t s) {
    if (B <= 0) return PD_OK;
    KlArgs a;
    a.N = op->N;
    a.N2 = op2 ? op2->N : 0;
    a.K = op->K;
    a.Kp = op->Kp;
    a.B = B;
    
    a.n_first = (a.N + kKlM - 1) / kKlM;
    a.n_tiles = a.n_first + (a.N2 + kKlM - 1) / kKlM;
    a.nt = pick_nt(a.n_tiles, B, op->Kp, op->sms);
    a.nbt = (B + a.nt - 1) / a.nt;
    a.marginal = marginal;
    a.mu = (float)mu;
    a.sig = (float)sig;
    a.wscale = (float)wscale;
    a.winvm = (float)winvm;
    a.xi = xi;
    a.out = out;
    a.out2 = out2;
    a.err = op->err;
    PD_REQUIRE(a.n_tiles * a.nbt < (1ll << 31), "too many KL tiles for one launch");
    // CTAs of a node tile's sample tiles are neighbours, so they read its Psi
    // rows together (once from DRAM); as many stages as fit
    const size_t smem_max = kKlSmem;
    a.stages = (int)std::min<size_t>(kKlStages, (smem_max - kl_smem_bytes(a.nt, op->Kp, 0)) / (2 * kKlM * 128));
    const size_t smem = kl_smem_bytes(a.nt, op->Kp, a.stages);
    const long long per = std::min<long long>(a.n_tiles, std::max<long long>(1, op->sms / a.nbt));
    k_sample_tc<<<(unsigned)(a.nbt * per), kKlThreads, smem, s>>>(op->tm, op2 ? op2->tm : op->tm, a);
    PD_CHECK_LAUNCH();
    return PD_OK;
}
