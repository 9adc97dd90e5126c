// pd_stencil.cu -- host side of the compile-time stencil step (the 122-offset
// horizon |k|^2 <= 9 of m in [3, sqrt(10)), and the 28-offset planar horizon
// of one-layer grids): the damage-slot layout and its maps to and from CSR
// order, the gather records, launch configuration and dispatch. The kernel
// itself is in pd_stencil_kernel.cuh.
#include <algorithm>
#include <cmath>
#include <cstdlib>
#include <mutex>
#include <utility>
#include <vector>

#include "pd_stencil_kernel.cuh"

namespace pdi {

namespace {

// Slot of node i, stencil code (2 m + t), in the per-sample damage array:
// [brick][warp][quad m / 4][lane][m % 4].
__device__ __forceinline__ long long slot_of(int i, int code, int nx, int ny, int BY, int BZ, int nbx, int nby,
                                             int wpb, int rounds) {
    const int ix = i % nx, iy = (i / nx) % ny, iz = i / (nx * ny);
    const long long brick = (ix / kSlice) + (long long)nbx * ((iy / BY) + (long long)nby * (iz / BZ));
    const int row = (iy % BY) + BY * (iz % BZ);
    const int w = row >> 1, rr = row & 1, c = ix % kSlice;
    const int m = code >> 1, t = code & 1;
    return (((brick * wpb + w) * (rounds / 4) + m / 4) * 32 + (16 * t + 8 * rr + c)) * 4 + (m % 4);
}

// Gather records of both parities from the state's double-float records:
// (u / dx rounded to FP32, s0 / 2), and the same point-reflected (node i of a
// sample at N - 1 - i).
__global__ void k_stencil_grec(long long N, long long NB, const float4 *rec0, const float4 *rec1, df idx, float4 *g0,
                               float4 *g1, float4 *r0, float4 *r1) {
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= NB) return;
    const long long b = t / N, i = t - b * N;
    for (int p = 0; p < 2; ++p) {
        const float4 *rc = p ? rec1 : rec0;
        const float4 h = rc[t], l = rc[NB + t];
        const float4 o = make_float4(df_mul(df{h.x, l.x}, idx).hi, df_mul(df{h.y, l.y}, idx).hi,
                                     df_mul(df{h.z, l.z}, idx).hi, 0.5f * h.w);
        (p ? g1 : g0)[t] = o;
        (p ? r1 : r0)[b * N + (N - 1 - i)] = o;
    }
}

// code of the CSR neighbour j of i: 2 m + t, or -1 if not a stencil offset
__device__ __forceinline__ int code_of(const int32_t *coord, int i, int j, const int16_t *box) {
    const int ci = coord[i], cj = coord[j];
    const int dx = (cj & 2047) - (ci & 2047), dy = ((cj >> 11) & 2047) - ((ci >> 11) & 2047), dz = (cj >> 22) - (ci >> 22);
    if (dx < -3 || dx > 3 || dy < -3 || dy > 3 || dz < -3 || dz > 3) return -1;
    return box[(dz + 3) * 49 + (dy + 3) * 7 + (dx + 3)];
}

// Damage template: 0 for every slot of a CSR bond, 1 (absent bond) elsewhere.
__global__ void k_stencil_template(const int32_t *row_ptr, const int32_t *col, const int32_t *coord, long long N,
                                   int nx, int ny, int BY, int BZ, int nbx, int nby, int wpb, int rounds,
                                   const int16_t *box, float *tmpl, int32_t *bad) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N) return;
    for (int p = row_ptr[i]; p < row_ptr[i + 1]; ++p) {
        const int code = code_of(coord, (int)i, col[p], box);
        if (code < 0) {
            bad[0] = 1;
            continue;
        }
        if (p > row_ptr[i] && col[p] <= col[p - 1]) bad[1] = 1;  // rows not in ascending order
        tmpl[slot_of((int)i, code, nx, ny, BY, BZ, nbx, nby, wpb, rounds)] = 0.0f;
    }
}

__global__ void k_fill_float(float *p, long long n, float v) {
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t < n) p[t] = v;
}

// Damage of every sample from the template, four words a thread (bound by the
// writes; 28k nodes x 32 samples, GB300: 71 us, 239 us one word at a time).
__global__ void __launch_bounds__(256) k_stencil_reset(long long len4, int B, const float4 *tmpl, float4 *dmg) {
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= len4) return;
    const float4 v = tmpl[t];
    for (int b = blockIdx.y; b < B; b += gridDim.y) __stcs(dmg + (size_t)b * len4 + t, v);
}

// FP32 to FP64 with integer operations: conversions run on the FP64 pipe (2
// lanes an SM on this part), which would bound a copy of 10^8 damage words.
// Zero and normal numbers only; the rest takes the conversion.
__device__ __forceinline__ double widen(float x) {
    const uint32_t u = __float_as_uint(x), e = (u >> 23) & 0xffu;
    if (u << 1 == 0u) return __hiloint2double((int)u, 0);
    if (e == 0u || e == 255u) return (double)x;
    return __hiloint2double((int)((u & 0x80000000u) | (((u & 0x7fffffffu) >> 3) + 0x38000000u)), (int)(u << 29));
}

// Damage between the stencil layout and CSR order (FP64). A warp takes the 16
// nodes of a row pair, for several samples: its 32 lanes' words go through
// shared memory so that both sides move whole lines. A CSR row lists the
// bonds of sub-lane 1 (offsets -k_m) by descending round, then those of
// sub-lane 0 (+k_m) by ascending round; the template says which exist. Both
// directions are bound by the memory they move and its latency (28k nodes x 32 samples, GB300:
// store 131 to 170 us, load 344 us; one thread per node and row, every word at a
// stride: 1,311 and 931 us).
//  * Storing reads only the groups of rounds that a sample has changed (dirty);
//    a row pair without any writes zeros.
//  * Loading also sets the dirty bits: a group of 8 rounds whose loaded damage
//    is not all zero is marked, in the byte of the part of the half-stencil
//    that owns it (q parts; bit group - first group of the part).
constexpr int kMapWarps = 4;
template <int DIM, bool TO_STATE>
__global__ void __launch_bounds__(32 * kMapWarps, 6) k_stencil_map(const int32_t *row_ptr, int B, long long nb, int nx,
                                                                int ny, int nz, int BY, int BZ, int nbx, int nby,
                                                                int wpb, long long n_rp, const float4 *tmpl,
                                                                float4 *dmg, double *csr, uint32_t *dirty, int q) {
    constexpr int R = Sten<DIM>::kRounds, H = Sten<DIM>::kHalf, G = R / 8;
    __shared__ float s_w[kMapWarps][32][R + 1];
    __shared__ uint32_t s_d[kMapWarps][32];  // loading: the lanes' dirty bits
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const long long rp = (long long)blockIdx.x * kMapWarps + warp;  // row pair: brick, then pair
    if (rp >= n_rp) return;
    float(*w)[R + 1] = s_w[warp];
    // present bonds of this lane, by round
    unsigned long long pm = 0ull;
    const float4 *tq = tmpl + rp * (R / 4) * 32 + lane;
#pragma unroll
    for (int g = 0; g < R / 4; ++g) {
        const float4 v = tq[32 * g];
        pm |= (unsigned long long)((v.x == 0.f ? 1u : 0u) | (v.y == 0.f ? 2u : 0u) | (v.z == 0.f ? 4u : 0u) |
                                   (v.w == 0.f ? 8u : 0u))
              << (4 * g);
    }
    const int brick = (int)(rp / wpb), row0 = 2 * (int)(rp % wpb);
    const int x0 = kSlice * (brick % nbx), by0 = BY * ((brick / nbx) % nby), bz0 = BZ * (brick / (nbx * nby));
    const int nv = min(kSlice, nx - x0), gpp = G / q;
    const long long len4 = n_rp * (R / 4) * 32;
    for (int b = blockIdx.y; b < B; b += gridDim.y) {
        float4 *dq = dmg + (size_t)b * len4 + rp * (R / 4) * 32 + lane;
        uint32_t *dw = dirty + ((size_t)b * n_rp + rp) * 32 + lane;
        bool zero = false;  // storing: no word of the row pair differs from the template
        if (!TO_STATE) {
            const uint32_t d = *dw;
            zero = !__any_sync(0xffffffffu, d != 0u);
            if (!zero) {
#pragma unroll
                for (int g = 0; g < G; ++g) {
                    const bool own = (d >> (8 * (g / gpp) + g % gpp)) & 1u;
                    float4 v0 = make_float4(0.f, 0.f, 0.f, 0.f), v1 = v0;
                    if (own) {
                        v0 = dq[64 * g];
                        v1 = dq[64 * g + 32];
                    }
                    float *o = &w[lane][8 * g];
                    o[0] = v0.x, o[1] = v0.y, o[2] = v0.z, o[3] = v0.w;
                    o[4] = v1.x, o[5] = v1.y, o[6] = v1.z, o[7] = v1.w;
                }
            }
        } else {
#pragma unroll
            for (int m = 0; m < R; ++m)  // absent bonds stay broken
                w[lane][m] = ((m < 32 ? (uint32_t)pm : (uint32_t)(pm >> 32)) >> (m % 32)) & 1u ? 0.f : 1.f;
            s_d[warp][lane] = 0u;
        }
        __syncwarp();
        for (int r = 0; r < 2; ++r) {
            const int row = row0 + r, gy = by0 + row % BY, gz = bz0 + row / BY;
            if (gy >= ny || gz >= nz) continue;  // warp-uniform
            const long long i0 = x0 + (long long)nx * (gy + (long long)ny * gz);
            if (!TO_STATE && zero) {  // the rows of a slice are contiguous
                double *o = csr + (size_t)b * nb;
                for (int e = row_ptr[i0] + lane; e < row_ptr[i0 + nv]; e += 32) __stcs(o + e, 0.0);
                continue;
            }
            for (int c = 0; c < nv; ++c) {
                const int l0 = 8 * r + c;
                const unsigned long long p1 = __shfl_sync(0xffffffffu, pm, l0 + 16), p0 = __shfl_sync(0xffffffffu, pm, l0);
                const int n1 = __popcll(p1);
                double *o = csr + (size_t)b * nb + row_ptr[i0 + c];
                // this lane's positions lane, lane + 32, ...: word (nullptr: absent) and CSR place
                constexpr int E = (2 * H + 31) / 32;
                float *word[E];
                double v[E];
                int at[E];
#pragma unroll
                for (int q4 = 0; q4 < E; ++q4) {
                    const int e = 32 * q4 + lane;
                    const bool neg = e < H;
                    const int m = neg ? H - 1 - e : e - H;
                    const unsigned long long p = neg ? p1 : p0;
                    const bool in = e < 2 * H && ((p >> m) & 1ull);
                    word[q4] = in ? &w[neg ? l0 + 16 : l0][m] : nullptr;
                    at[q4] = neg ? __popcll(p >> 1 >> m) : n1 + __popcll(p & ((1ull << m) - 1ull));
                }
                if (TO_STATE) {
#pragma unroll
                    for (int q4 = 0; q4 < E; ++q4) v[q4] = word[q4] ? __ldcs(o + at[q4]) : 0.0;
#pragma unroll
                    for (int q4 = 0; q4 < E; ++q4)  // (an integer test: FP64 compares run on the FP64 pipe)
                        if (__double_as_longlong(v[q4]) << 1) {
                            const float f = (float)v[q4];
                            const int at_w = (int)(word[q4] - &w[0][0]), l = at_w / (R + 1), g = at_w % (R + 1) / 8;
                            *word[q4] = f;
                            if (f != 0.f) atomicOr(&s_d[warp][l], 1u << (8 * (g / gpp) + g % gpp));
                        }
                } else {
#pragma unroll
                    for (int q4 = 0; q4 < E; ++q4)
                        if (word[q4]) __stcs(o + at[q4], widen(*word[q4]));
                }
            }
        }
        __syncwarp();
        if (TO_STATE) {
#pragma unroll
            for (int g = 0; g < G; ++g) {
                const float *o = &w[lane][8 * g];
                __stcs(dq + 64 * g, make_float4(o[0], o[1], o[2], o[3]));
                __stcs(dq + 64 * g + 32, make_float4(o[4], o[5], o[6], o[7]));
            }
            *dw = s_d[warp][lane];
            __syncwarp();
        }
    }
}

// The same for a neighbour list whose rows are not in ascending order (any
// order of a row's neighbours is accepted): one thread per node. Loading (TO_STATE)
// also sets the damage flags of the node's two lanes: a group of 8 rounds
// whose loaded damage is not all zero (the template value of a present bond)
// is marked, in the byte of the part of the half-stencil that owns it (q
// parts; byte part of the lane's word, bit group - first group of the part).
// A node's bonds lie in its own two lanes only, so each word has one writer.
template <bool TO_STATE>
__global__ void k_stencil_map_any(const int32_t *row_ptr, const int32_t *col, const int32_t *coord, long long N, int B,
                              long long nb, int nx, int ny, int BY, int BZ, int nbx, int nby, int wpb, int rounds,
                              long long len, const int16_t *box, float *dmg, double *csr, uint32_t *dirty,
                              int q) {
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= N * B) return;
    const int b = (int)(t / N);
    const int i = (int)(t % N);
    const int gpp = rounds / 8 / q;  // groups of 8 rounds per part
    uint32_t w[2] = {0u, 0u};        // flags of sub-lanes 0 and 1
    for (int p = row_ptr[i]; p < row_ptr[i + 1]; ++p) {
        const int code = code_of(coord, i, col[p], box);
        if (code < 0) continue;
        const long long e = (long long)b * len + slot_of(i, code, nx, ny, BY, BZ, nbx, nby, wpb, rounds);
        const long long qq = (long long)b * nb + p;
        if (TO_STATE) {
            const float d = (float)csr[qq];
            dmg[e] = d;
            if (d != 0.0f) {
                const int g = (code >> 1) / 8, part = g / gpp;
                w[code & 1] |= 1u << (8 * part + (g - part * gpp));
            }
        } else {
            csr[qq] = (double)dmg[e];
        }
    }
    if (TO_STATE) {
        const int ix = i % nx, iy = (i / nx) % ny, iz = i / (nx * ny);
        const long long brick = (ix / kSlice) + (long long)nbx * ((iy / BY) + (long long)nby * (iz / BZ));
        const int row = (iy % BY) + BY * (iz % BZ);
        const long long lane0 = (brick * wpb + (row >> 1)) * 32 + 8 * (row & 1) + (ix % kSlice);
        const long long per_sample = len / rounds;  // lanes of a sample
        dirty[(size_t)b * per_sample + lane0] = w[0];
        dirty[(size_t)b * per_sample + lane0 + 16] = w[1];
    }
}

// Slot, in one sample's damage array, of every CSR bond (every CSR neighbour
// is a stencil offset: checked when the template is built).
__global__ void k_stencil_slots(const int32_t *row_ptr, const int32_t *col, const int32_t *coord, long long N,
                                int nx, int ny, int BY, int BZ, int nbx, int nby, int wpb, int rounds,
                                const int16_t *box, long long *slot) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N) return;
    for (int p = row_ptr[i]; p < row_ptr[i + 1]; ++p) {
        const int code = code_of(coord, (int)i, col[p], box);
        slot[p] = code < 0 ? 0 : slot_of((int)i, code, nx, ny, BY, BZ, nbx, nby, wpb, rounds);
    }
}

// Warps of 16 nodes (100 for each of the part's 152 SMs); the line lies between
// the two sizes measured, 10,240 (slower) and 22,400 (faster): see one_lane.
constexpr long long kOneLanePairs = 152ll * 100;

StencilPairFn pick_pair(int dim, int q, int law, bool kappa) {
    if (dim == 2) return stencil_pair_d2(law, kappa);
    if (q == 4) return stencil_pair_d3q4(law, kappa);
    if (q == 2) return stencil_pair_d3q2(law, kappa);
    return stencil_pair_d3q1(law, kappa);
}

// The step kernel variant of a launch (force-only evaluations take the
// one-sample kernel).
StencilKernel pick_stencil(int dim, int ns, int q, int law, bool kappa, bool fo) {
    if (dim == 2) return stencil_pick_d2(ns, law, kappa, fo);  // 16 rounds: two groups of 8 at Q = 1 only
    if (q == 4) return stencil_pick_d3q4(ns, law, kappa, fo);
    if (q == 2) return stencil_pick_d3q2(ns, law, kappa, fo);
    return stencil_pick_d3q1(ns, law, kappa, fo);
}

// One lane per node for plane launches whose warps of 32 nodes fill the GPU
// (pairs: both meshes' blocks together): a plane node has 14 rounds per role,
// so the set-up and the integration weigh more than the bonds (89,600 nodes x 4
// samples, GB300: 28.1 us a step against 32.1). With fewer nodes, two lanes
// per node keep more warps in flight (10,240 warps of 16 nodes: 17.5 us with one
// lane, 15.7 with two). In 3D (61 rounds) it is slower: 160
// against 152 us for an elastic step of the 28k-node beam x 32, and 248 against
// 217 ms for a run to the peak, where a warp meets twice the fix-ups.
bool one_lane(const pd_state *st, long long row_pairs) {
    return st->st_dim == 2 && st->st_ns == 1 && st->st_q == 1 && st->st_wpb % 2 == 0 && st->st_wpb <= 8 &&
           row_pairs >= kOneLanePairs;
}

unsigned blocks_of(long long n) { return (unsigned)((n + 255) / 256); }

}  // namespace

// Dynamic shared memory of a launch: the upper and the reflected lower copy
// of the staged records (BZ + halo layers each), the same for kappa when a
// stiffness field is set, and the partial sums of Q > 1 parts.
// Dynamic shared memory of a launch: the two record copies, each rounded up to
// 128 bytes (TMA destinations), the kappa copies, the parts' partial sums,
// and 128 bytes to align the box.
size_t stencil_smem(const pd_state *st, int ns, bool kappa) {
    const int hz = st->st_dim == 3 ? Sten<3>::kHaloZ : Sten<2>::kHaloZ;
    const size_t rows = (size_t)(st->by + 2 * kHalo) * (st->bz + hz);
    size_t b = 2 * ((rows * ns * kRowC + 127) & ~(size_t)127) + 128;
    if (kappa) b += 2 * rows * ns * kRowK;
    return b + (size_t)(st->st_q - 1) * st->st_wpb * 16 * 6 * ns * sizeof(float);
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static EncodeTiledFn tiled_encoder() {
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

// Map of a [B][nz][ny][nx] array of 4-float records, read in boxes of 14 cells
// x Wy rows x Zp layers of one sample; cells outside the grid read as zero.
static int encode_box_map(CUtensorMap *tm, float4 *base, const pd_state *st, int Wy, int Zp) {
    EncodeTiledFn enc = tiled_encoder();
    PD_REQUIRE(enc != nullptr, "cuTensorMapEncodeTiled is unavailable");
    const cuuint64_t nx = (cuuint64_t)st->g.nx, ny = (cuuint64_t)st->g.ny, nz = (cuuint64_t)st->g.nz;
    const cuuint64_t dims[5] = {4, nx, ny, nz, (cuuint64_t)st->B};
    const cuuint64_t strides[4] = {16, 16 * nx, 16 * nx * ny, 16 * nx * ny * nz};
    const cuuint32_t box[5] = {4, (cuuint32_t)kWx, (cuuint32_t)Wy, (cuuint32_t)Zp, 1};
    const cuuint32_t estr[5] = {1, 1, 1, 1, 1};
    const CUresult r = enc(tm, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 5, base, dims, strides, box, estr,
                           CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                           CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    PD_REQUIRE(r == CUDA_SUCCESS, "cuTensorMapEncodeTiled failed for the stencil box (%d)", (int)r);
    return PD_OK;
}

bool stencil_applicable(const pd_state *st) {
    const double m2 = st->g.m_ratio * st->g.m_ratio;
    return st->mat.precision == PD_PREC_MIXED && m2 >= 9.0 && m2 < 10.0 && ((st->by * st->bz) % 2 == 0) &&
           st->by * st->bz <= 32;
}

// The dynamic shared-memory limit of the stencil kernels only ever grows (per
// device): states of several meshes coexist (the fine and coarse members of
// MLMC pairs) and each launches with its own brick size.
int stencil_set_attributes(size_t smem) {
    static std::mutex mu;
    static size_t limit[64] = {};
    int dev = 0;
    PD_CHECK_CUDA(cudaGetDevice(&dev));
    std::lock_guard<std::mutex> lock(mu);
    if (dev >= 0 && dev < 64 && smem <= limit[dev]) return PD_OK;
    for (int dim = 2; dim <= 3; ++dim)
        for (int ns = 1; ns <= 2; ++ns)
            for (int q = 1; q <= 4; q *= 2)
                for (int law = 0; law < 2; ++law)
                    for (int kap = 0; kap < 2; ++kap)
                        for (int fo = 0; fo < 2; ++fo)
                            PD_CHECK_CUDA(cudaFuncSetAttribute((const void *)pick_stencil(dim, ns, q, law, kap, fo),
                                                               cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                               (int)smem));
    for (int dim = 2; dim <= 3; ++dim)
        for (int q = 1; q <= 4; q *= 2)
            for (int law = 0; law < 2; ++law)
                for (int kap = 0; kap < 2; ++kap)
                    PD_CHECK_CUDA(cudaFuncSetAttribute((const void *)pick_pair(dim, q, law, kap),
                                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    for (int law = 0; law < 2; ++law)
        for (int kap = 0; kap < 2; ++kap) {
            const void *one[2] = {(const void *)stencil_pick_d2_1l(law, kap), (const void *)stencil_pair_d2_1l(law, kap)};
            for (const void *k : one)
                PD_CHECK_CUDA(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        }
    if (dev >= 0 && dev < 64) limit[dev] = smem;
    return PD_OK;
}

int stencil_build(pd_state *st, const int32_t *col) {
    const long long N = st->N;
    st->st_wpb = st->by * st->bz / 2;
    st->st_dim = st->g.nz == 1 ? 2 : 3;  // a one-layer grid has only the planar offsets
    const int rounds = st->st_dim == 3 ? Sten<3>::kRounds : Sten<2>::kRounds;
    st->st_len = st->n_bricks * st->st_wpb * (long long)rounds * 32;
    // samples per block: one (measured on GB300, a pair per block is slower at
    // 122 registers a thread, 16 warps per SM); pairs on request
    st->st_ns = st->ns_req ? st->ns_req : 1;
    // split the half-stencil over Q warps when the mesh gives too few warps per SM
    // (measured on GB300: Q = 2 for single samples of the 28k-node beam, 1 for batches)
    const long long warps1 = st->n_bricks * ((st->B + st->st_ns - 1) / st->st_ns) * st->st_wpb;
    st->st_q = warps1 >= 152ll * 24 ? 1 : 2;
    if (st->q_req) st->st_q = st->q_req;
    if (st->st_dim == 2) st->st_q = 1;
    // threads a block: at most 512, or 256 for one sample at Q = 2 (its register budget)
    while (st->st_q > 1 && 32 * st->st_wpb * st->st_q > (st->st_q == 2 && st->st_ns == 1 ? 256 : 512)) st->st_q /= 2;
    // Deferring the reaction to the next launch pays when a launch is a
    // single wave of a few blocks per SM, whose reduction tail would
    // otherwise stand alone at the end (measured on GB300: 28k-node beam,
    // one sample, 19.3 -> 18 us per step); with many waves the tail overlaps
    // other blocks and the deferred read only adds to each block's start.
    {
        int dev = 0, sms = 0;
        PD_CHECK_CUDA(cudaGetDevice(&dev));
        PD_CHECK_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
        st->st_one_wave = st->n_bricks * ((st->B + st->st_ns - 1) / st->st_ns) <= 4ll * sms;
        st->st_defer = st->st_one_wave;
        if (st->reduce_req) st->st_defer = st->reduce_req == 2;
    }
    // the largest launch of this state (kappa staged; force-only evaluations
    // take the one-sample kernel, which needs no more)
    st->smem_bytes = stencil_smem(st, st->st_ns, true);
    PD_REQUIRE(st->smem_bytes <= 227 * 1024, "stencil brick 8x%dx%d for %d samples needs %zu bytes of shared memory",
               st->by, st->bz, st->st_ns, st->smem_bytes);
    std::vector<int16_t> box(343, -1);
    const int half = st->st_dim == 3 ? Sten<3>::kHalf : Sten<2>::kHalf;
    for (int m = 0; m < half; ++m) {
        const I3 k = st->st_dim == 3 ? half_off<3>(m) : half_off<2>(m);
        box[(k.z + 3) * 49 + (k.y + 3) * 7 + (k.x + 3)] = (int16_t)(2 * m);
        box[(-k.z + 3) * 49 + (-k.y + 3) * 7 + (-k.x + 3)] = (int16_t)(2 * m + 1);
    }
    PD_TRY(dalloc(&st->st_box, box.size()));
    PD_CHECK_CUDA(cudaMemcpy(st->st_box, box.data(), box.size() * sizeof(int16_t), cudaMemcpyHostToDevice));
    PD_TRY(dalloc(&st->st_tmpl, st->st_len));
    PD_TRY(dalloc(&st->st_dirty, (size_t)st->B * (st->st_len / rounds) * 4));
    PD_CHECK_CUDA(cudaMemset(st->st_dirty, 0, (size_t)st->B * (st->st_len / rounds) * 4));
    PD_TRY(dalloc(&st->grec[0], (size_t)st->B * N));
    PD_TRY(dalloc(&st->grec[1], (size_t)st->B * N));
    PD_TRY(dalloc(&st->grecR[0], (size_t)st->B * N));
    PD_TRY(dalloc(&st->grecR[1], (size_t)st->B * N));
    {
        const int Wy = st->by + 2 * kHalo;
        const int Zp = st->bz + (st->st_dim == 3 ? Sten<3>::kHaloZ : Sten<2>::kHaloZ);
        for (int p = 0; p < 2; ++p) {
            PD_TRY(encode_box_map(&st->st_maps.rec[p], st->grec[p], st, Wy, Zp));
            PD_TRY(encode_box_map(&st->st_maps.ref[p], st->grecR[p], st, Wy, Zp));
        }
    }
    // every slot starts as an absent (broken) bond; the slots of real bonds are cleared
    k_fill_float<<<blocks_of(st->st_len), 256>>>(st->st_tmpl, st->st_len, 1.0f);
    PD_CHECK_LAUNCH();
    int32_t *bad = nullptr;
    PD_TRY(dalloc(&bad, 2));
    cudaMemset(bad, 0, 2 * sizeof(int32_t));
    k_stencil_template<<<blocks_of(N), 256>>>(st->row_ptr, col, st->coord, N, st->g.nx, st->g.ny, st->by, st->bz,
                                              st->nbx, st->nby, st->st_wpb, rounds, st->st_box, st->st_tmpl, bad);
    int32_t hbad[2] = {0, 0};
    const cudaError_t e = cudaMemcpy(hbad, bad, sizeof(hbad), cudaMemcpyDeviceToHost);
    cudaFree(bad);
    PD_CHECK_CUDA(e);
    PD_REQUIRE(!hbad[0], "a CSR neighbour is not a horizon stencil offset of the grid");
    st->st_sorted = hbad[1] == 0;
    return stencil_set_attributes(st->smem_bytes);
}

int stencil_refresh_grec(pd_state *st, cudaStream_t s) {
    const long long NB = st->N * st->B;
    k_stencil_grec<<<blocks_of(NB), 256, 0, s>>>(st->N, NB, (const float4 *)st->rec[0], (const float4 *)st->rec[1],
                                                 df_split(1.0 / st->g.dx), st->grec[0], st->grec[1], st->grecR[0],
                                                 st->grecR[1]);
    PD_CHECK_LAUNCH();
    return PD_OK;
}

void stencil_fill_args(const pd_state *st, StepArgs &a) {
    a.grec0 = st->grec[0];
    a.grec1 = st->grec[1];
    a.grecR0 = st->grecR[0];
    a.grecR1 = st->grecR[1];
    a.idx_df = df_split(1.0 / st->g.dx);
    a.tmpl = st->st_tmpl;
    a.dirty = st->st_dirty;
    a.fd_grp1 = fastdiv_make(st->B);
    a.fd_grp2 = fastdiv_make((st->B + 1) / 2);
    a.fd_nbx = fastdiv_make(st->nbx);
    a.fd_nby = fastdiv_make(st->nby);
    a.fd_by = fastdiv_make(st->by);
}

// Samples that a block of a per-state pass takes in turn: as few as give the
// pass about 16 blocks an SM.
static unsigned sample_blocks(const pd_state *st, long long blocks_x) {
    return (unsigned)std::max<long long>(1, std::min<long long>(st->B, (152 * 16 + blocks_x - 1) / blocks_x));
}

int stencil_reset_damage(pd_state *st, cudaStream_t s) {
    const unsigned gx = blocks_of(st->st_len / 4);
    k_stencil_reset<<<dim3(gx, sample_blocks(st, gx)), 256, 0, s>>>(st->st_len / 4, st->B, (const float4 *)st->st_tmpl,
                                                                   (float4 *)st->dmg);
    PD_CHECK_LAUNCH();
    // every group equals the template again
    const int rounds = st->st_dim == 3 ? Sten<3>::kRounds : Sten<2>::kRounds;
    PD_CHECK_CUDA(cudaMemsetAsync(st->st_dirty, 0, (size_t)st->B * (st->st_len / rounds) * 4, s));
    return PD_OK;
}

int stencil_map_damage(const pd_state *st, double *csr, bool to_state, cudaStream_t s) {
    if (!st->st_sorted) {
        const auto any = to_state ? k_stencil_map_any<true> : k_stencil_map_any<false>;
        any<<<blocks_of(st->N * st->B), 256, 0, s>>>(
            st->row_ptr, st->col_csr, st->coord, st->N, st->B, st->nb, st->g.nx, st->g.ny, st->by, st->bz, st->nbx,
            st->nby, st->st_wpb, st->st_dim == 3 ? Sten<3>::kRounds : Sten<2>::kRounds, st->st_len, st->st_box,
            (float *)st->dmg, csr, (uint32_t *)st->st_dirty, st->st_q);
        PD_CHECK_LAUNCH();
        return PD_OK;
    }
    const long long n_rp = st->n_bricks * st->st_wpb;
    const unsigned gx = (unsigned)((n_rp + kMapWarps - 1) / kMapWarps);
    const auto k = st->st_dim == 3 ? (to_state ? k_stencil_map<3, true> : k_stencil_map<3, false>)
                                   : (to_state ? k_stencil_map<2, true> : k_stencil_map<2, false>);
    k<<<dim3(gx, sample_blocks(st, gx)), 32 * kMapWarps, 0, s>>>(
        st->row_ptr, st->B, st->nb, st->g.nx, st->g.ny, st->g.nz, st->by, st->bz, st->nbx, st->nby, st->st_wpb, n_rp,
        (const float4 *)st->st_tmpl, (float4 *)st->dmg, csr, (uint32_t *)st->st_dirty, st->st_q);
    PD_CHECK_LAUNCH();
    return PD_OK;
}

int stencil_slot_table(const pd_state *st, long long *slot, cudaStream_t s) {
    k_stencil_slots<<<blocks_of(st->N), 256, 0, s>>>(st->row_ptr, st->col_csr, st->coord, st->N, st->g.nx, st->g.ny,
                                                     st->by, st->bz, st->nbx, st->nby, st->st_wpb,
                                                     st->st_dim == 3 ? Sten<3>::kRounds : Sten<2>::kRounds,
                                                     st->st_box, slot);
    PD_CHECK_LAUNCH();
    return PD_OK;
}

bool stencil_pairable(const pd_state *s0, const pd_state *s1) {
    return s0->stencil && s1->stencil && s0->st_ns == 1 && s1->st_ns == 1 && s0->st_dim == s1->st_dim &&
           s0->st_q == s1->st_q && s0->st_wpb == s1->st_wpb && s0->mat.law == s1->mat.law &&
           s0->has_kappa == s1->has_kappa;
}

// A step launch of many waves may start while the previous kernel in the
// stream is finishing (programmatic dependent launch): the kernel waits for it
// (griddepcontrol.wait) before it reads anything, so only the launch and the
// scheduling of its blocks overlap the previous step's tail. Single-wave
// launches (one sample of a small mesh) are launched plainly: there the
// steps without softening gain (28k-node beam, one sample, GB300: 12.4 ->
// 10.8 us) but the steps with a growing crack lose more, and whole runs to
// the peak were slower (14.07 against 14.00 us per step).
static cudaLaunchConfig_t pdl_config(unsigned grid, int threads, size_t smem, cudaStream_t s, bool pdl) {
    static const cudaLaunchAttribute attr = [] {
        cudaLaunchAttribute x{};
        x.id = cudaLaunchAttributeProgrammaticStreamSerialization;
        x.val.programmaticStreamSerializationAllowed = 1;
        return x;
    }();
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = const_cast<cudaLaunchAttribute *>(&attr);
    cfg.numAttrs = pdl ? 1 : 0;
    return cfg;
}

int stencil_launch_pair(const pd_state *s0, const StepArgs &a0, const pd_state *s1, const StepArgs &a1,
                        cudaStream_t s) {
    PD_REQUIRE(stencil_pairable(s0, s1), "the two states do not share a launch shape");
    StepPair g;
    g.a[0] = a0;
    g.a[1] = a1;
    g.nblk0 = (int)s0->n_bricks * s0->B;
    g.t[0] = s0->st_maps;
    g.t[1] = s1->st_maps;
    const unsigned grid = (unsigned)g.nblk0 + (unsigned)s1->n_bricks * (unsigned)s1->B;
    const size_t smem = std::max(stencil_smem(s0, 1, s0->has_kappa), stencil_smem(s1, 1, s1->has_kappa));
    const bool one = one_lane(s0, (long long)grid * s0->st_wpb);
    const StencilPairFn k = !one ? pick_pair(s0->st_dim, s0->st_q, s0->mat.law, s0->has_kappa)
                                : stencil_pair_d2_1l(s0->mat.law, s0->has_kappa);
    cudaLaunchConfig_t cfg = pdl_config(grid, (one ? 16 : 32) * s0->st_wpb * s0->st_q, smem, s,
                                        !s0->st_one_wave || !s1->st_one_wave);
    PD_CHECK_CUDA(cudaLaunchKernelEx(&cfg, k, g));
    return PD_OK;
}

int stencil_launch(const pd_state *st, const StepArgs &a, bool force_only, cudaStream_t s) {
    const int ns = force_only ? 1 : st->st_ns;
    const unsigned grid = (unsigned)st->n_bricks * (unsigned)((st->B + ns - 1) / ns);
    const bool one = !force_only && one_lane(st, (long long)grid * st->st_wpb);
    StencilKernel k = !one ? pick_stencil(st->st_dim, ns, st->st_q, st->mat.law, st->has_kappa, force_only)
                          : stencil_pick_d2_1l(st->mat.law, st->has_kappa);
    cudaLaunchConfig_t cfg =
        pdl_config(grid, (one ? 16 : 32) * st->st_wpb * st->st_q, stencil_smem(st, ns, st->has_kappa), s, !st->st_one_wave);
    PD_CHECK_CUDA(cudaLaunchKernelEx(&cfg, k, a, st->st_maps));
    return PD_OK;
}

}  // namespace pdi
