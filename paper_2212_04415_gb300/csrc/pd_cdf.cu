// pd_cdf.cu -- multilevel estimate of the peak-load distribution (Section 7):
// the inverse CDF F_L^-1(u) = R_0^[N_0 u] + sum_{l >= 1} (R_l^[N_l u] -
// R~_{l-1}^[N_l u]), where R_l are the fine and R~_{l-1} the coarse members of
// level l's pairs, each sorted ascending, and R^[k] is the k-th smallest.
// Readings: the index [N u] is ceil(N u), 1-based, clamped to [1, N]; the
// coarse term of level l uses the level's own pair count N_l (with N_{l-1},
// as printed, the sum would telescope to the finest level alone). The CDF at
// x is the fraction of the points F_L^-1((i + 1/2) / n), i < n, that are <= x.
//
// Every level's members are sorted stably (equal values, -0 and +0 among them,
// keep their order): tiles of 1,024 in shared memory, then merge passes of up
// to 32 sorted runs in which each element finds its place by one binary search
// per run. All arrays of a call (fine and coarse members of every
// level) share each launch, so a call of 20,000 + 3,000 + 300 samples is two
// launches. Values compare as integers of the same order: FP64 compares run on
// the narrow FP64 pipe of this part (2 lanes an SM). Measured on GB300, one
// pd_ml_inverse_cdf and one pd_ml_cdf of that size through the Python binding:
// 0.23 to 0.26 ms; an exact rank count of every element against all others took
// 8.3 to 8.6 ms.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <utility>

#include "pd_internal.cuh"

namespace pdi {

constexpr int kSortTile = 1024;  // elements sorted by one block
constexpr int kSortFan = 32;     // runs merged by one pass
constexpr int kMaxSegs = 2 * PD_MAX_LEVELS;

// The arrays of one call. Element e of the call lies in segment q with
// off[q] <= e < off[q] + n[q]; every buffer of the call has this layout.
struct SortSegs {
    int n_segs;
    long long n[kMaxSegs], off[kMaxSegs];
    long long tile0[kMaxSegs];  // first tile of the segment (tiles do not cross segments)
    const double *src[kMaxSegs];
};

// Integer of the same order as the value (-0 and +0 equal).
__device__ __forceinline__ unsigned long long order_key(double v) {
    const unsigned long long top = 1ull << 63;
    unsigned long long b = (unsigned long long)__double_as_longlong(v);
    if (b == top) b = 0ull;
    return (b & top) ? ~b : (b | top);
}

// One tile: bitonic sort of (key, position) pairs, one in the registers of
// each thread; positions break ties, so the order is stable. One wave of blocks
// at MLMC sample counts, bound by the latency of its 55 exchanges: the 40 of
// distance 16 or less are shuffles, the other 15 pass through shared memory
// (two buffers in turn, so each costs one barrier). All 55 in shared memory, two
// elements a thread: 14.7 us against 12.3 (ncu, 28 tiles).
__global__ void __launch_bounds__(kSortTile) k_sort_tiles(const SortSegs g, double *out) {
    __shared__ unsigned long long s_key[2][kSortTile];
    __shared__ int s_pos[2][kSortTile];
    int q = 0;
    while (q + 1 < g.n_segs && (long long)blockIdx.x >= g.tile0[q + 1]) ++q;
    const long long e0 = ((long long)blockIdx.x - g.tile0[q]) * kSortTile;
    const int m = (int)min((long long)kSortTile, g.n[q] - e0);
    const double *x = g.src[q] + e0;
    const int i = threadIdx.x;
    unsigned long long key = i < m ? order_key(x[i]) : ~0ull;
    int pos = i, buf = 0;
    const auto keep = [&](unsigned long long k2, int p2, bool smaller) {
        const bool other_less = k2 < key || (k2 == key && p2 < pos);
        if (other_less == smaller) {
            key = k2;
            pos = p2;
        }
    };
    for (int k = 2; k <= kSortTile; k <<= 1) {
        for (int j = k >> 1; j > 0; j >>= 1) {
            const bool smaller = ((i & j) == 0) == ((i & k) == 0);
            if (j >= 32) {
                s_key[buf][i] = key;
                s_pos[buf][i] = pos;
                __syncthreads();
                keep(s_key[buf][i ^ j], s_pos[buf][i ^ j], smaller);
                buf ^= 1;
            } else {
                const unsigned long long k2 = __shfl_xor_sync(0xffffffffu, key, j);
                const int p2 = __shfl_xor_sync(0xffffffffu, pos, j);
                keep(k2, p2, smaller);
            }
        }
    }
    if (pos < m) out[g.off[q] + e0 + i] = x[pos];
}

// One merge pass: sorted runs of `run` elements, kSortFan of them to a group,
// become one run each. A block places 32 elements: its warps share the runs of
// the group, each lane counting the elements of a run that go before its own
// element. The lanes' elements are neighbours, so their searches read the same
// lines (a lane per run and a warp per element: 21 us against 12, ncu,
// 26,600 elements in 20 + 3 + 3 + 1 + 1 runs). The padding elements of a tile
// are all last (their key is the largest and their position beyond every real
// one), so no run holds any.
constexpr int kMergeWarps = 8;
__global__ void __launch_bounds__(32 * kMergeWarps) k_merge_runs(const SortSegs g, long long total, long long run,
                                                                 int runs, const double *in, double *out) {
    __shared__ long long s_before[kMergeWarps][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const long long w = (long long)blockIdx.x * 32 + lane;
    const bool ok = w < total;
    const long long e = ok ? w : total - 1;
    int q = 0;
    while (q + 1 < g.n_segs && e >= g.off[q + 1]) ++q;
    const double *x = in + g.off[q];
    const long long i = e - g.off[q], n = g.n[q];
    const long long group = run * kSortFan, g0 = i / group * group;
    const int own = (int)((i - g0) / run);
    const double v = x[i];
    const unsigned long long kv = order_key(v);
    long long before = 0;
    for (int r = warp; r < runs; r += kMergeWarps) {
        const long long lo0 = g0 + r * run, hi0 = min(n, lo0 + run);
        if (r == own) {
            before += i - lo0;
        } else if (lo0 < hi0) {  // r < own: elements <= v go first; r > own: elements < v
            long long lo = lo0, hi = hi0;
            while (lo < hi) {
                const long long mid = (lo + hi) >> 1;
                const unsigned long long km = order_key(x[mid]);
                if (km < kv || (km == kv && r < own))
                    lo = mid + 1;
                else
                    hi = mid;
            }
            before += lo - lo0;
        }
    }
    s_before[warp][lane] = before;
    __syncthreads();
    if (warp == 0 && ok) {
#pragma unroll
        for (int o = 1; o < kMergeWarps; ++o) before += s_before[o][lane];
        out[g.off[q] + g0 + before] = v;
    }
}

struct CdfLevels {
    int n_levels;
    long long n[PD_MAX_LEVELS];
    long long off[PD_MAX_LEVELS];
};

__device__ __forceinline__ long long order_index(long long N, double u) {
    long long k = (long long)ceil((double)N * u);
    k = k < 1 ? 1 : (k > N ? N : k);
    return k - 1;
}

__device__ __forceinline__ double ml_inverse(const CdfLevels &L, const double *sf, const double *sc, double u) {
    double v = sf[L.off[0] + order_index(L.n[0], u)];
    for (int l = 1; l < L.n_levels; ++l) {
        const long long k = order_index(L.n[l], u);
        v += sf[L.off[l] + k] - sc[L.off[l] + k];
    }
    return v;
}

__global__ void k_ml_inverse(CdfLevels L, const double *sf, const double *sc, int n_u, const double *u,
                             double *out) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t < n_u) out[t] = ml_inverse(L, sf, sc, u[t]);
}

__global__ void k_ml_points(CdfLevels L, const double *sf, const double *sc, int n_u, double *X) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t < n_u) X[t] = ml_inverse(L, sf, sc, ((double)t + 0.5) / (double)n_u);
}

// One warp per x: its lanes share the points.
__global__ void __launch_bounds__(256) k_cdf_count(int n_u, const double *X, int n_x, const double *x, double *F) {
    const int t = (int)(((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
    if (t >= n_x) return;  // warp-uniform
    const double xt = x[t];
    int c = 0;
#pragma unroll 8
    for (long long i = lane; i < n_u; i += 32) c += X[i] <= xt ? 1 : 0;
    c = __reduce_add_sync(0xffffffffu, c);
    if (lane == 0) F[t] = (double)c / (double)n_u;
}

// Sorted fine and coarse members of every level (level-major, as given): sf
// and sc point into buf, which also holds `extra` doubles at *rest.
static int sort_levels(int n_levels, const int64_t *n_per_level, const double *q_fine, const double *q_coarse,
                       CdfLevels &L, Scratch &buf, const double *&sf, const double *&sc, long long extra,
                       double *&rest, cudaStream_t s) {
    PD_REQUIRE(n_levels >= 1 && n_levels <= PD_MAX_LEVELS, "n_levels out of range");
    PD_REQUIRE(n_per_level && q_fine, "n_per_level and q_fine are required");
    PD_REQUIRE(n_levels == 1 || q_coarse, "q_coarse is required with more than one level");
    long long tot = 0, longest = 0;
    L.n_levels = n_levels;
    for (int l = 0; l < n_levels; ++l) {
        PD_REQUIRE(n_per_level[l] >= 1, "every level needs at least one sample");
        L.n[l] = n_per_level[l];
        L.off[l] = tot;
        tot += n_per_level[l];
        longest = std::max(longest, L.n[l]);
    }
    // the fine members at [0, tot), the coarse members of levels 1, 2, ... at
    // [tot, 2 tot - n_0) with the same spacing
    SortSegs g;
    memset(&g, 0, sizeof(g));
    long long tiles = 0;
    for (int m = 0; m < 2; ++m)
        for (int l = m; l < n_levels; ++l) {
            const int q = g.n_segs++;
            g.n[q] = L.n[l];
            g.off[q] = m == 0 ? L.off[l] : tot + L.off[l] - L.off[1];
            g.src[q] = (m ? q_coarse : q_fine) + L.off[l];
            g.tile0[q] = tiles;
            tiles += (L.n[l] + kSortTile - 1) / kSortTile;
        }
    const long long all = g.off[g.n_segs - 1] + g.n[g.n_segs - 1];
    PD_TRY(scratch_alloc(buf, (size_t)(2 * all + extra) * sizeof(double), s));
    double *a = (double *)buf.p, *b = a + all;
    rest = a + 2 * all;
    k_sort_tiles<<<(unsigned)tiles, kSortTile, 0, s>>>(g, a);
    PD_CHECK_LAUNCH();
    for (long long run = kSortTile; run < longest; run *= kSortFan) {
        const long long runs = std::min<long long>((longest + run - 1) / run, kSortFan);
        k_merge_runs<<<(unsigned)((all + 31) / 32), 32 * kMergeWarps, 0, s>>>(g, all, run, (int)runs, a, b);
        PD_CHECK_LAUNCH();
        std::swap(a, b);
    }
    sf = a;
    sc = n_levels > 1 ? a + tot - L.off[1] : nullptr;  // indexed with the levels' offsets
    return PD_OK;
}

}  // namespace pdi

using namespace pdi;

extern "C" int pd_ml_inverse_cdf(int32_t n_levels, const int64_t *n_per_level, const double *q_fine,
                                 const double *q_coarse, int32_t n_u, const double *u, double *out,
                                 pd_stream stream) {
    PD_REQUIRE(n_u >= 0 && (n_u == 0 || (u && out)), "u and out are required");
    cudaStream_t s = (cudaStream_t)stream;
    CdfLevels L;
    Scratch buf;
    const double *sf, *sc;
    double *rest;
    PD_TRY(sort_levels(n_levels, n_per_level, q_fine, q_coarse, L, buf, sf, sc, 0, rest, s));
    if (n_u) {
        k_ml_inverse<<<(n_u + 255) / 256, 256, 0, s>>>(L, sf, sc, n_u, u, out);
        PD_CHECK_LAUNCH();
    }
    PD_CHECK_CUDA(cudaStreamSynchronize(s));
    return PD_OK;
}

extern "C" int pd_ml_cdf(int32_t n_levels, const int64_t *n_per_level, const double *q_fine,
                         const double *q_coarse, int32_t n_u, int32_t n_x, const double *x, double *F,
                         pd_stream stream) {
    PD_REQUIRE(n_u >= 1, "n_u must be >= 1");
    PD_REQUIRE(n_x >= 0 && (n_x == 0 || (x && F)), "x and F are required");
    cudaStream_t s = (cudaStream_t)stream;
    CdfLevels L;
    Scratch buf;
    const double *sf, *sc;
    double *X;
    PD_TRY(sort_levels(n_levels, n_per_level, q_fine, q_coarse, L, buf, sf, sc, n_u, X, s));
    k_ml_points<<<(n_u + 255) / 256, 256, 0, s>>>(L, sf, sc, n_u, X);
    PD_CHECK_LAUNCH();
    if (n_x) {
        k_cdf_count<<<(unsigned)(((long long)n_x * 32 + 255) / 256), 256, 0, s>>>(n_u, X, n_x, x, F);
        PD_CHECK_LAUNCH();
    }
    PD_CHECK_CUDA(cudaStreamSynchronize(s));
    return PD_OK;
}
