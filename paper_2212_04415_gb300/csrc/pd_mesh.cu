// pd_mesh.cu -- neighbour list (horizon, Eq. PD_Horizon) and boundary sets.
//
// The grid is regular, so the horizon of a node is a fixed integer stencil
// |offset|^2 <= m^2 (in cell units) clipped by the body and by the notch
// plane. Rows list their neighbours in ascending linear index order, so the
// list is a pure integer function of the grid (bit-exact, no atomics).
//
// Four launches (grid of 448,000 nodes, 50M bonds, GB300, count and fill calls
// together with their three host synchronisations: 0.24 ms; with one thread
// walking a node's candidate box for both passes and a one-block scan of every
// row: 4.6 ms):
//   k_row_counts  a thread per node counts whole x-ranges of the stencil's
//                 (dy, dz) rows, beside the notch, whose cut does not depend on
//                 z, whole z-ranges of its (dx, dy) columns (16 us; with candidates
//                 one by one there 23.5), and its block leaves running sums;
//   k_scan_ends   one block scans the last element of every 256;
//   k_add_ends    the other elements get their block's start;
//   k_fill_rows   a warp per node writes the row, 32 neighbours at a time
//                 (bound by the writes, 4 bytes a bond).
#include <stdarg.h>
#include <string.h>

#include <algorithm>
#include <cmath>

#include "pd_internal.cuh"

namespace pdi {

static thread_local char g_err[512] = "";

void set_error(const char *fmt, ...) {
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(g_err, sizeof(g_err), fmt, ap);
    va_end(ap);
}

int validate_grid(const pd_grid *g) {
    PD_REQUIRE(g != nullptr, "grid is NULL");
    PD_REQUIRE(g->nx > 0 && g->ny > 0 && g->nz > 0, "grid sizes must be positive");
    PD_REQUIRE(g->nx <= 2047 && g->ny <= 2047 && g->nz <= 1023,
               "grid too large for packed coordinates (nx, ny <= 2047, nz <= 1023)");
    PD_REQUIRE((int64_t)g->nx * g->ny * g->nz < (1ll << 31), "more than 2^31 nodes");
    PD_REQUIRE(g->dx > 0.0 && std::isfinite(g->dx), "dx must be positive");
    PD_REQUIRE(g->m_ratio > 0.0 && g->m_ratio <= 8.0, "m_ratio must be in (0, 8]");
    return PD_OK;
}

constexpr int kMaxR = 8;  // largest offset component (m_ratio <= 8)

struct GridDev {
    int nx, ny, nz, r;  // r: largest offset component
    int notch, X2, Y2;
    int all;            // neighbours of a node away from the faces and the notch
    signed char hw[2 * kMaxR * kMaxR + 1];  // largest dx >= 0 with dx^2 + q <= m^2 (-1: none), q = dy^2 + dz^2
};

// Strict crossing of the notch plane below the tip, in exact integers.
__device__ __forceinline__ bool notch_cut(const GridDev &g, int ix, int iy, int jx, int jy) {
    if (!g.notch) return false;
    const long long Xi = 2 * ix + 1, Xj = 2 * jx + 1;
    const long long Yi = 2 * iy + 1, Yj = 2 * jy + 1;
    const long long Xn = g.X2;
    if ((Xi - Xn) * (Xj - Xn) >= 0) return false;
    const long long dX = Xj - Xi;
    const long long lhs = Yi * dX + (Xn - Xi) * (Yj - Yi);
    const long long rhs = (long long)g.Y2 * dX;
    return dX > 0 ? (lhs < rhs) : (lhs > rhs);
}

constexpr int kMeshBlock = 256;
constexpr int kMaxOff = 2108;    // offsets with 0 < |k|^2 <= 64
constexpr int kMaxWords = (kMaxOff + 31) / 32;
constexpr int kFillNodes = 8;    // consecutive nodes a warp fills at a time (one load of their row starts)

// Near the notch: some bond of a node at (ix, iy) may cross the plane (within
// a horizon of it in x) below its tip (its lower end reaches below the tip).
__device__ __forceinline__ bool near_notch(const GridDev &g, int ix, int iy) {
    return g.notch && llabs(2ll * ix + 1 - g.X2) <= 2 * g.r && 2ll * (iy - g.r) + 1 < g.Y2;
}

// row_ptr[i + 1] = neighbours of the nodes of i's block up to i.
__global__ void __launch_bounds__(kMeshBlock) k_row_counts(const __grid_constant__ GridDev g, int32_t *__restrict__ row_ptr) {
    __shared__ int wsum[kMeshBlock / 32];
    const long long n = (long long)g.nx * g.ny * g.nz;
    const long long i = (long long)blockIdx.x * kMeshBlock + threadIdx.x;
    int cnt = 0;
    if (i < n) {
        const int ix = (int)((unsigned)i % (unsigned)g.nx), yz = (int)((unsigned)i / (unsigned)g.nx);
        const int iy = (int)((unsigned)yz % (unsigned)g.ny), iz = (int)((unsigned)yz / (unsigned)g.ny);
        const bool cut = near_notch(g, ix, iy);
        if (!cut && ix >= g.r && ix < g.nx - g.r && iy >= g.r && iy < g.ny - g.r && iz >= g.r && iz < g.nz - g.r) {
            cnt = g.all;
        } else {
            if (!cut) {
                for (int dz = max(-g.r, -iz); dz <= min(g.r, g.nz - 1 - iz); ++dz)
                    for (int dy = max(-g.r, -iy); dy <= min(g.r, g.ny - 1 - iy); ++dy) {
                        const int h = g.hw[dy * dy + dz * dz];
                        cnt += max(min(ix + h, g.nx - 1) - max(ix - h, 0) + 1, 0);
                    }
            } else {  // whether the notch cuts a bond does not depend on z
                for (int dy = max(-g.r, -iy); dy <= min(g.r, g.ny - 1 - iy); ++dy)
                    for (int dx = max(-g.r, -ix); dx <= min(g.r, g.nx - 1 - ix); ++dx) {
                        const int h = g.hw[dx * dx + dy * dy];
                        if (h >= 0 && !notch_cut(g, ix, iy, ix + dx, iy + dy))
                            cnt += min(h, iz) + min(h, g.nz - 1 - iz) + 1;
                    }
            }
            --cnt;  // the node itself (never cut) is not its neighbour
        }
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int v = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += u;
    }
    if (lane == 31) wsum[warp] = v;
    __syncthreads();
    for (int w = 0; w < warp; ++w) v += wsum[w];
    if (i < n) row_ptr[i + 1] = v;
    if (i == 0) row_ptr[0] = 0;
}

// Inclusive scan of the block ends row_ptr[min(256 (b + 1), n)] in place, one
// block; totals past 2^31 - 1 are clamped and flagged. out: total, overflow.
__global__ void __launch_bounds__(1024) k_scan_ends(int32_t *a, long long n, long long nblk, int32_t *out) {
    __shared__ long long part[32];
    const int t = threadIdx.x;
    const long long per = (nblk + 1023) / 1024;
    const long long lo = min(nblk, t * per), hi = min(nblk, lo + per);
    const auto end = [&](long long b) { return min((b + 1) * kMeshBlock, n); };
    long long s = 0;
    for (long long b = lo; b < hi; ++b) s += a[end(b)];
    // inclusive scan of the 1024 partial sums: within warps, then over warps
    const int lane = t & 31, warp = t >> 5;
    const auto warp_scan = [&](long long v) {
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const long long u = __shfl_up_sync(0xffffffffu, v, o);
            if (lane >= o) v += u;
        }
        return v;
    };
    long long v = warp_scan(s);
    if (lane == 31) part[warp] = v;
    __syncthreads();
    if (warp == 0) part[lane] = warp_scan(part[lane]);
    __syncthreads();
    if (warp > 0) v += part[warp - 1];
    long long run = v - s;
    for (long long b = lo; b < hi; ++b) {
        run += a[end(b)];
        a[end(b)] = (int32_t)min(run, 2147483647ll);
    }
    if (t == 1023) {
        out[0] = (int32_t)min(v, 2147483647ll);
        out[1] = v > 2147483647ll ? 1 : 0;
    }
}

__global__ void __launch_bounds__(kMeshBlock) k_add_ends(int32_t *a, long long n) {
    const long long b0 = ((long long)blockIdx.x + 1) * kMeshBlock;  // this block's start, from block 1 on
    const long long k = b0 + 1 + threadIdx.x;
    if (k < min(b0 + kMeshBlock, n)) a[k] = (int32_t)min((long long)a[k] + a[b0], 2147483647ll);
}

// The rows of a horizon of at most 32 NW offsets (NW = 0: any). Blocks list the stencil's offsets in shared memory (ascending
// linear order), with masks of the offsets that stay inside for every distance
// of a node from each face; then their warps take nodes in turn: a node away
// from the faces and the notch writes every offset, others compact 32 offsets
// at a time by the masks (beside the notch after an exact test as well). With
// NW = 4 (128 offsets: horizons below 3.17 cells) the offsets and the masks of
// the current row of nodes stay in registers (85 us on the 448,000-node beam);
// the loops over any number of words take 103 us there.
template <int NW>
__global__ void __launch_bounds__(kMeshBlock) k_fill_rows(const __grid_constant__ GridDev g,
                                                          const int32_t *__restrict__ row_ptr,
                                                          int32_t *__restrict__ col) {
    __shared__ int s_lin[kMaxOff];
    __shared__ int s_k[kMaxOff];
    __shared__ unsigned s_in[6][kMaxR + 1][kMaxWords];  // [face x0 x1 y0 y1 z0 z1][distance][word]
    __shared__ int s_w[kMeshBlock / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int D = 2 * g.r + 1;
    int n_off = 0;
    for (int q0 = 0; q0 < D * D * D; q0 += kMeshBlock) {
        const int q = q0 + threadIdx.x;
        const int dx = q % D - g.r, dy = (q / D) % D - g.r, dz = q / (D * D) - g.r;
        const bool cell = q < D * D * D;
        const bool in = cell && abs(dx) <= g.hw[cell ? dy * dy + dz * dz : 0] && (dx || dy || dz);
        const unsigned m = __ballot_sync(0xffffffffu, in);
        if (lane == 0) s_w[warp] = __popc(m);
        __syncthreads();
        int at = n_off + __popc(m & ((1u << lane) - 1u));
        for (int w = 0; w < kMeshBlock / 32; ++w) {
            if (w < warp) at += s_w[w];
            n_off += s_w[w];
        }
        if (in) {
            s_lin[at] = dx + g.nx * (dy + g.ny * dz);
            s_k[at] = (dx & 0xff) | ((dy & 0xff) << 8) | ((dz & 0xff) << 16);
        }
        __syncthreads();
    }
    const int n_words = (n_off + 31) / 32;
    for (int t = warp; t < 6 * (g.r + 1) * n_words; t += kMeshBlock / 32) {
        const int w = t % n_words, e = t / n_words % (g.r + 1), f = t / n_words / (g.r + 1);
        const int q = 32 * w + lane;
        // offset away from the lower (f even) or the upper face, at distance e from it
        const int k = q < n_off ? (int)(signed char)((s_k[q] >> (8 * (f / 2))) & 0xff) : 0;
        const unsigned m = __ballot_sync(0xffffffffu, q < n_off && (f & 1 ? k <= e : k >= -e));
        if (lane == 0) s_in[f][e][w] = m;
    }
    __syncthreads();
    constexpr int RW = NW ? NW : 1;
    int lin[RW];
    unsigned zy[RW];
    if (NW) {
#pragma unroll
        for (int w = 0; w < RW; ++w) lin[w] = 32 * w + lane < n_off ? s_lin[32 * w + lane] : 0;
    }
    const long long n = (long long)g.nx * g.ny * g.nz;
    const long long step = (long long)gridDim.x * (kMeshBlock / 32) * kFillNodes;
    for (long long i0 = ((long long)blockIdx.x * (kMeshBlock / 32) + warp) * kFillNodes; i0 < n; i0 += step) {
        const int m_nodes = (int)min((long long)kFillNodes, n - i0);
        const int base = lane < m_nodes ? row_ptr[i0 + lane] : 0;
        int ix = (int)((unsigned)i0 % (unsigned)g.nx);
        const int yz = (int)((unsigned)i0 / (unsigned)g.nx);
        int iy = (int)((unsigned)yz % (unsigned)g.ny), iz = (int)((unsigned)yz / (unsigned)g.ny);
        bool new_row = true;
        const unsigned *y0 = nullptr, *y1 = nullptr, *z0 = nullptr, *z1 = nullptr;
        for (int c = 0; c < m_nodes; ++c) {
            if (new_row) {
                y0 = s_in[2][min(iy, g.r)];
                y1 = s_in[3][min(g.ny - 1 - iy, g.r)];
                z0 = s_in[4][min(iz, g.r)];
                z1 = s_in[5][min(g.nz - 1 - iz, g.r)];
                if (NW) {
#pragma unroll
                    for (int w = 0; w < RW; ++w) zy[w] = w < n_words ? y0[w] & y1[w] & z0[w] & z1[w] : 0u;
                }
                new_row = false;
            }
            const int i = (int)i0 + c;
            int32_t *out = col + __shfl_sync(0xffffffffu, base, c);
            const unsigned *x0 = s_in[0][min(ix, g.r)], *x1 = s_in[1][min(g.nx - 1 - ix, g.r)];
            const bool xin = ix >= g.r && ix < g.nx - g.r, cut = near_notch(g, ix, iy);
            const auto put = [&](int w, unsigned m, int lw) {
                const int q = 32 * w + lane;
                if (!xin) m &= x0[w] & x1[w];
                if (cut) {  // warp-uniform
                    const int k = q < n_off ? s_k[q] : 0;
                    m &= ~__ballot_sync(0xffffffffu, notch_cut(g, ix, iy, ix + (int)(signed char)(k & 0xff),
                                                               iy + (int)(signed char)((k >> 8) & 0xff)));
                }
                if ((m >> lane) & 1u) out[__popc(m & ((1u << lane) - 1u))] = i + lw;
                out += __popc(m);
            };
            if (NW) {
#pragma unroll
                for (int w = 0; w < RW; ++w) put(w, zy[w], lin[w]);
            } else {
                for (int w = 0; w < n_words; ++w)
                    put(w, y0[w] & y1[w] & z0[w] & z1[w], 32 * w + lane < n_off ? s_lin[32 * w + lane] : 0);
            }
            if (++ix == g.nx) {
                ix = 0;
                new_row = true;
                if (++iy == g.ny) {
                    iy = 0;
                    ++iz;
                }
            }
        }
    }
}

static GridDev make_dev(const pd_grid *g) {
    GridDev d = {};
    d.nx = g->nx;
    d.ny = g->ny;
    d.nz = g->nz;
    const double m2 = g->m_ratio * g->m_ratio;
    d.r = 0;
    while (d.r < kMaxR && (double)((d.r + 1) * (d.r + 1)) <= m2) ++d.r;
    for (int q = 0; q <= 2 * d.r * d.r; ++q) {
        int h = -1;
        while (h < d.r && (double)((h + 1) * (h + 1) + q) <= m2) ++h;
        d.hw[q] = (signed char)h;
    }
    d.all = -1;  // the node itself is no neighbour
    for (int dz = -d.r; dz <= d.r; ++dz)
        for (int dy = -d.r; dy <= d.r; ++dy) d.all += 2 * d.hw[dy * dy + dz * dz] + 1 > 0 ? 2 * d.hw[dy * dy + dz * dz] + 1 : 0;
    d.notch = g->notch ? 1 : 0;
    d.X2 = g->notch_x2;
    d.Y2 = g->notch_y2;
    return d;
}

__global__ void k_bc(int nx, int ny, int nz, pd_bc bc, uint8_t *__restrict__ codes) {
    const long long n = (long long)nx * ny * nz;
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int ix = (int)(i % nx), iy = (int)((i / nx) % ny);
    const int X = 2 * ix + 1;
    uint8_t c0 = 0, c1 = 0, c2 = 0;
    if (bc.type == PD_BC_BAR_TENSION) {
        if (ix < bc.grip_planes) {
            c0 = c1 = c2 = 1;
        } else if (ix >= nx - bc.grip_planes) {
            c0 = 2;
            c1 = c2 = 1;
        }
    } else {
        if (iy == 0) {
            const int d0 = X - bc.support_x2[0], d1 = X - bc.support_x2[1];
            if ((d0 >= -1 && d0 <= 1) || (d1 >= -1 && d1 <= 1)) c1 = 1;
        }
        if (iy == ny - 1) {
            const int d = X - bc.load_x2;
            if (d >= -1 && d <= 1) c1 = 3;
        }
    }
    codes[3 * i + 0] = c0;
    codes[3 * i + 1] = c1;
    codes[3 * i + 2] = c2;
}

}  // namespace pdi

using namespace pdi;

extern "C" int pd_last_error(char *buf, size_t len) {
    if (!buf || len == 0) return PD_ERR_ARG;
    strncpy(buf, g_err, len - 1);
    buf[len - 1] = 0;
    return PD_OK;
}

extern "C" const char *pd_version(void) { return "pd-gb300 0.1 (sm_103a)"; }

// row_ptr, the bond count and, with col, the rows; out2: two words of device
// scratch. Where calls in flight together share those (shared), the count, which
// the rows' space is checked against, comes from the caller's own row_ptr, so
// that no more than the overflow flag can be lost.
static int build_rows(const pd_grid *g, int32_t *row_ptr, int32_t *col, int64_t cap, int64_t *n_bonds, int32_t *out2,
                      bool shared, cudaStream_t s) {
    const long long n = (long long)g->nx * g->ny * g->nz;
    const long long nblk = (n + kMeshBlock - 1) / kMeshBlock;
    const GridDev d = make_dev(g);
    k_row_counts<<<(unsigned)nblk, kMeshBlock, 0, s>>>(d, row_ptr);
    PD_CHECK_LAUNCH();
    k_scan_ends<<<1, 1024, 0, s>>>(row_ptr, n, nblk, out2);
    PD_CHECK_LAUNCH();
    if (nblk > 1) {
        k_add_ends<<<(unsigned)(nblk - 1), kMeshBlock, 0, s>>>(row_ptr, n);
        PD_CHECK_LAUNCH();
    }
    int32_t h[2] = {0, 0};
    PD_CHECK_CUDA(cudaMemcpyAsync(h, out2, sizeof(h), cudaMemcpyDeviceToHost, s));
    int32_t total = 0;
    if (shared) PD_CHECK_CUDA(cudaMemcpyAsync(&total, row_ptr + n, sizeof(total), cudaMemcpyDeviceToHost, s));
    PD_CHECK_CUDA(cudaStreamSynchronize(s));
    if (!shared) total = h[0];
    PD_REQUIRE(!h[1], "more than 2^31-1 bonds");
    *n_bonds = total;
    if (col == nullptr) return PD_OK;
    if (cap < total) {
        set_error("col capacity %lld < %d bonds", (long long)cap, total);
        return PD_ERR_CAP;
    }
    int dev = 0, sms = 0;
    PD_CHECK_CUDA(cudaGetDevice(&dev));
    PD_CHECK_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    const long long per_blk = kMeshBlock / 32 * kFillNodes, need = (n + per_blk - 1) / per_blk;
    const auto fill = d.all <= 128 ? k_fill_rows<4> : k_fill_rows<0>;
    fill<<<(unsigned)std::min<long long>(need, 8ll * sms), kMeshBlock, 0, s>>>(d, row_ptr, col);
    PD_CHECK_LAUNCH();
    PD_CHECK_CUDA(cudaStreamSynchronize(s));  // the list is complete on return, for any stream
    return PD_OK;
}

extern "C" int pd_build_neighbours(const pd_grid *g, int32_t *row_ptr, int32_t *col, int64_t cap,
                                   int64_t *n_bonds, pd_stream stream) {
    PD_TRY(validate_grid(g));
    PD_REQUIRE(row_ptr != nullptr && n_bonds != nullptr, "row_ptr and n_bonds are required");
    cudaStream_t s = (cudaStream_t)stream;
    Scratch two;
    PD_TRY(scratch_alloc(two, 2 * sizeof(int32_t), s));
    return build_rows(g, row_ptr, col, cap, n_bonds, (int32_t *)two.p, false, s);
}

extern "C" int pd_bc_codes(const pd_grid *g, const pd_bc *bc, uint8_t *codes, pd_stream stream) {
    PD_TRY(validate_grid(g));
    PD_REQUIRE(bc != nullptr && codes != nullptr, "bc and codes are required");
    PD_REQUIRE(bc->type == PD_BC_BAR_TENSION || bc->type == PD_BC_BEAM_3PT, "unknown bc type %d", bc->type);
    const long long n = (long long)g->nx * g->ny * g->nz;
    k_bc<<<(unsigned)((n + 255) / 256), 256, 0, (cudaStream_t)stream>>>(g->nx, g->ny, g->nz, *bc, codes);
    PD_CHECK_LAUNCH();
    return PD_OK;
}

// ---------------------------------------------------------------------------
// Allocation-free variant of pd_build_neighbours.
//
// The build needs two words of device scratch beyond its inputs and outputs:
// the total of the row-pointer scan and its overflow flag. pd_build_neighbours
// takes them from the scratch pool on every call; this variant keeps them in a
// file-scope device array instead, for callers that cannot allocate device
// memory, and reads the total from row_ptr. The array's address is
// looked up on every call with the current device (cudaGetSymbolAddress), so a
// context torn down by cudaDeviceReset leaves no stale pointer behind.
static __device__ __align__(256) int32_t g_noalloc_scratch[64];  // 256 bytes; words 0 and 1: total, overflow

static int noalloc_scratch(int32_t **out) {
    void *p = nullptr;
    const cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
    if (e != cudaSuccess) {
        set_error("cudaGetSymbolAddress of the neighbour-build scratch failed: %s", cudaGetErrorString(e));
        return PD_ERR_CUDA;
    }
    *out = (int32_t *)p;
    return PD_OK;
}

extern "C" int pd_build_neighbours_noalloc(const pd_grid *g, int32_t *row_ptr, int32_t *col, int64_t cap,
                                           int64_t *n_bonds, pd_stream stream) {
    PD_TRY(validate_grid(g));
    PD_REQUIRE(row_ptr != nullptr && n_bonds != nullptr, "row_ptr and n_bonds are required");
    const long long n = (long long)g->nx * g->ny * g->nz;
    PD_REQUIRE(n + 1 <= 2147483647ll, "at most 2^31 - 2 nodes");
    cudaStream_t s = (cudaStream_t)stream;
    if (s != nullptr) {  // the scratch address is the current device's: the stream must run there
        int cur = 0, sdev = 0;
        PD_CHECK_CUDA(cudaGetDevice(&cur));
        PD_CHECK_CUDA(cudaStreamGetDevice(s, &sdev));
        PD_REQUIRE(sdev == cur, "the stream belongs to device %d, not the current device %d", sdev, cur);
    }
    int32_t *two = nullptr;
    PD_TRY(noalloc_scratch(&two));
    return build_rows(g, row_ptr, col, cap, n_bonds, two, true, s);  // both words are written on every call
}
