// pd_adjoint_stencil.cu -- the adjoint run of mixed-path states on the
// compile-time stencil (the recursion stated in pd_adjoint.cu), in the
// stencil's own layout:
//
//  * Checkpoints are the state's arrays as they are (records, velocities,
//    damage words, dirty bits): plain copies, no passage through CSR order.
//  * Damage never decreases, so a bond whose final damage equals its initial
//    one keeps it at every step and is never active. Two 128-bit masks per node
//    and sample, in the order of the node's CSR row over the full stencil, say
//    which bonds grow in the run and which others are damaged; the damage
//    trajectory and the damage adjoint (double-float) hold the growing bonds
//    only, node after node.
//  * The bond adjoint (k_adj_bonds_st) stages the node records (u, s0) and
//    (lamF, kappa) of a tile of nodes and its halo in shared memory and one
//    thread per node walks the node's row: the positions over the stencil are
//    bytes shared by the samples, offset, xi, |xi| and 1/|xi| come from a table
//    in shared memory, growing and damaged are mask bits. A node's terms are
//    summed in FP32 over 8 bonds at a time and folded into compensated sums
//    (fixed order: the row's), then added to the FP64 node sums; the integrator
//    adjoint of the step before follows in the same thread.
//
// 28k-node beam x 32 samples, stiffness field, GB300 (ncu): bond adjoint
// 430 us a step (644 us over a sliced-ELL copy of the rows, whose offsets,
// lengths and damage codes are loaded and decoded per bond); damage gather
// 16 us a step with the node records (85 us over all slots); a checkpoint
// is four copies, 1.1 GB moved (through CSR order: 1,311 us store and 931 us load). 60 steps with checkpoints
// every 20: 59.0 ms (98.4).
#include <algorithm>
#include <cmath>

#include "pd_stencil_kernel.cuh"

#include "pd_adjoint.cuh"

namespace pdi {

namespace {

// ------------------------------------------------------------ bond masks

// Position of a slot in its node's row over the full stencil: offsets -k_m by
// descending m, then +k_m.
template <int DIM>
__host__ __device__ constexpr int row_pos(int m, int t) {
    return t ? Sten<DIM>::kHalf - 1 - m : Sten<DIM>::kHalf + m;
}

// Brick layout of a state's damage words.
struct Lay {
    int nx, ny, nz, BY, BZ, nbx, nby, wpb;
    long long n_rp;  // row pairs
    long long N;
};

__device__ __forceinline__ unsigned long long widen_half(unsigned long long lo, unsigned long long hi, int sh,
                                                         unsigned long long &top) {
    top = hi >> (64 - sh);
    return lo | (hi << sh);
}

// Per node and sample: bonds that grow between d0 and d1 and bonds that keep a
// damage other than zero (masks over the node's CSR row), the count of the
// former; for sample 0 also the node's present bonds (over the full stencil). A warp per row pair and sample; only
// groups of damage that differ from the template at the end are read.
template <int DIM>
__global__ void __launch_bounds__(256) k_adj_masks(const Lay y, const float4 *tmpl, const float4 *d0, const float4 *d1,
                                                   const uint32_t *dirty1, int q, ulonglong2 *present,
                                                   ulonglong2 *grow, ulonglong2 *keep, long long *count) {
    constexpr int R = Sten<DIM>::kRounds, H = Sten<DIM>::kHalf, G = R / 8;
    const long long rp = (long long)blockIdx.x * 8 + (threadIdx.x >> 5);
    if (rp >= y.n_rp) return;
    const int lane = threadIdx.x & 31, b = blockIdx.y, t = lane >> 4;
    const size_t base = rp * (R / 4) * 32 + lane, samp = (size_t)b * y.n_rp * (R / 4) * 32;
    const int gpp = G / q;
    unsigned long long pm = 0ull, gm = 0ull, km = 0ull;  // by row position within the half
    const auto bit = [&](int m) { return 1ull << (t ? H - 1 - m : m); };
    const uint32_t dw = dirty1[((size_t)b * y.n_rp + rp) * 32 + lane];
    for (int g = 0; g < G; ++g) {
        const bool dirty = (dw >> (8 * (g / gpp) + g % gpp)) & 1u;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const float4 tv = tmpl[base + 32 * (2 * g + h)];
            float4 a = make_float4(0.f, 0.f, 0.f, 0.f), c = a;
            if (dirty) {
                a = d0[samp + base + 32 * (2 * g + h)];
                c = d1[samp + base + 32 * (2 * g + h)];
            }
            const float tw[4] = {tv.x, tv.y, tv.z, tv.w}, aw[4] = {a.x, a.y, a.z, a.w}, cw[4] = {c.x, c.y, c.z, c.w};
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int m = 8 * g + 4 * h + j;
                if (m >= H || tw[j] != 0.f) continue;  // absent
                pm |= bit(m);
                if (dirty && cw[j] > aw[j])
                    gm |= bit(m);
                else if (dirty && aw[j] != 0.f)
                    km |= bit(m);
            }
        }
    }
    // sub-lane 1's half is the low part of the row
    const auto row = [&](unsigned long long v) {
        const unsigned long long o = __shfl_xor_sync(0xffffffffu, v, 16);
        ulonglong2 r;
        r.x = widen_half(o, v, H, r.y);  // (on sub-lane 0: o = sub-lane 1's)
        return r;
    };
    const ulonglong2 P = row(pm), Gr = row(gm), Kp = row(km);
    // positions over the full stencil -> positions in the row
    const auto squeeze = [&](const ulonglong2 &v) {
        ulonglong2 r = make_ulonglong2(0ull, 0ull);
        const int n0 = __popcll(P.x);
        for (unsigned long long w = v.x; w; w &= w - 1) r.x |= 1ull << __popcll(P.x & ((w & -w) - 1));
        for (unsigned long long w = v.y; w; w &= w - 1) {
            const int at = n0 + __popcll(P.y & ((w & -w) - 1));
            (at < 64 ? r.x : r.y) |= 1ull << (at & 63);
        }
        return r;
    };
    const int brick = (int)(rp / y.wpb), rw = 2 * (int)(rp % y.wpb) + ((lane >> 3) & 1);
    const int gx = kSlice * (brick % y.nbx) + (lane & 7), gy = y.BY * ((brick / y.nbx) % y.nby) + rw % y.BY,
              gz = y.BZ * (brick / (y.nbx * y.nby)) + rw / y.BY;
    if (t == 0 && gx < y.nx && gy < y.ny && gz < y.nz) {
        const long long i = gx + (long long)y.nx * (gy + (long long)y.ny * gz);
        if (b == 0) present[i] = P;
        grow[(size_t)b * y.N + i] = squeeze(Gr);
        keep[(size_t)b * y.N + i] = squeeze(Kp);
        count[(size_t)b * y.N + i + 1] = __popcll(Gr.x) + __popcll(Gr.y);
    }
}

// Inclusive scan of a[1 .. n] (a[0] = 0): blocks of 1024, the block ends, the rest.
__global__ void __launch_bounds__(1024) k_scan64_blocks(long long *a, long long n) {
    __shared__ long long part[32];
    const long long i = (long long)blockIdx.x * 1024 + threadIdx.x;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    long long v = i < n ? a[i + 1] : 0;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const long long u = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += u;
    }
    if (lane == 31) part[warp] = v;
    __syncthreads();
    for (int w = 0; w < warp; ++w) v += part[w];
    if (i < n) a[i + 1] = v;
    if (i == 0) a[0] = 0;
}
__global__ void __launch_bounds__(1024) k_scan64_ends(long long *a, long long n, long long nblk) {
    __shared__ long long part[32];
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const long long per = (nblk + 1023) / 1024, lo = min(nblk, t * per), hi = min(nblk, lo + per);
    const auto end = [&](long long b) { return min((b + 1) * 1024, n); };
    const auto warp_scan = [&](long long v) {
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const long long u = __shfl_up_sync(0xffffffffu, v, o);
            if (lane >= o) v += u;
        }
        return v;
    };
    long long s = 0;
    for (long long b = lo; b < hi; ++b) s += a[end(b)];
    long long v = warp_scan(s);
    if (lane == 31) part[warp] = v;
    __syncthreads();
    if (warp == 0) part[lane] = warp_scan(part[lane]);
    __syncthreads();
    if (warp > 0) v += part[warp - 1];
    long long run = v - s;
    for (long long b = lo; b < hi; ++b) a[end(b)] = run += a[end(b)];
}
__global__ void __launch_bounds__(1024) k_scan64_add(long long *a, long long n) {
    const long long b0 = ((long long)blockIdx.x + 1) * 1024, k = b0 + 1 + threadIdx.x;
    if (k < min(b0 + 1024, n)) a[k] += a[b0];
}

// Damage word, within a sample, of the bond at row position e of node i.
template <int DIM>
__device__ __forceinline__ long long word_of(const Lay &y, int i, int e) {
    constexpr int R = Sten<DIM>::kRounds, H = Sten<DIM>::kHalf;
    const int ix = i % y.nx, iy = (i / y.nx) % y.ny, iz = i / (y.nx * y.ny);
    const long long brick = (ix / kSlice) + (long long)y.nbx * ((iy / y.BY) + (long long)y.nby * (iz / y.BZ));
    const int row = (iy % y.BY) + y.BY * (iz % y.BZ);
    const int t = e < H ? 1 : 0, m = t ? H - 1 - e : e - H;
    return (((brick * y.wpb + (row >> 1)) * (R / 4) + m / 4) * 32 + (16 * t + 8 * (row & 1) + ix % kSlice)) * 4 + m % 4;
}

// Damage words of the growing bonds, node after node in row order. W: 32 bits
// where a sample's words fit them, 64 above (from 2^25 node places of whole
// bricks on; every step reads the list).
template <int DIM, class W>
__global__ void __launch_bounds__(256) k_adj_list(const Lay y, int B, const ulonglong2 *present, const ulonglong2 *grow,
                                                  const long long *base, W *words) {
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= y.N * B) return;
    const ulonglong2 g = grow[t];
    if (!(g.x | g.y)) return;
    const int i = (int)(t % y.N);
    const ulonglong2 P = present[i];
    long long o = base[t];
    int r = 0;  // row position
    for (int h = 0; h < 2; ++h)
        for (unsigned long long w = h ? P.y : P.x; w; w &= w - 1, ++r)
            if (((r < 64 ? g.x : g.y) >> (r & 63)) & 1ull) words[o++] = (W)word_of<DIM>(y, i, 64 * h + __ffsll(w) - 1);
}

// The current records of the samples whose step has the other parity than n0
// (blockIdx.y: sample), into the buffer of n0's.
__global__ void __launch_bounds__(256) k_adj_align(long long N, long long BN, const int32_t *step, int n0, float4 *rec0,
                                                   float4 *rec1) {
    if (!((step[blockIdx.y] ^ n0) & 1)) return;
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N) return;
    const size_t t = (size_t)blockIdx.y * N + i;
    const float4 *from = n0 & 1 ? rec0 : rec1;
    float4 *to = n0 & 1 ? rec1 : rec0;
    to[t] = from[t];
    to[BN + t] = from[BN + t];
}

// The growing bonds' damage at the current step (blockIdx.y: sample) and, with
// rec, the node records (u, s0), u = u_hi + u_lo rounded to FP32.
template <class W>
__global__ void __launch_bounds__(256) k_adj_snap(long long N, long long BN, const long long *base, const W *words,
                                                  const float *dmg, long long st_len, float *out, const float4 *rec,
                                                  float4 *u4) {
    const int b = blockIdx.y;
    const float *src = dmg + (size_t)b * st_len;
    const long long g1 = base[(b + 1) * N], step = (long long)gridDim.x * blockDim.x;
    const long long t0 = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    for (long long x = base[b * N] + t0; x < g1; x += step) out[x] = __ldg(src + words[x]);
    if (rec) {
        for (long long i = t0; i < N; i += step) {
            const float4 h = rec[b * N + i], l = rec[BN + b * N + i];
            u4[b * N + i] = make_float4(h.x + l.x, h.y + l.y, h.z + l.z, h.w);
        }
    }
}

// --------------------------------------------------------- reverse sweep

// Integrator adjoint of local step `ls` at node i of sample b, from lamu^{n+1}
// (lu): lamv in place, and (lamF, kappa) in FP32 for the bond adjoint.
__device__ __forceinline__ float4 node_adjoint(const AdjArgs &a, int ls, long long i, int b, const double lu[3],
                                               double *lv) {
    float f[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const uint8_t code = a.codes[3 * i + c];
        double lF = 0.0, v = 0.0;
        if (code == 0) {
            const double lvp = lv[c] + a.dt * lu[c];
            lF = a.dt_rb * lvp;
            v = a.a_b * lvp;
        } else if (code != 1) {
            double wn = 0.0;
            for (int o = 0; o < a.n_obs; ++o)
                if (a.obs[o] == ls) wn += a.w[(size_t)b * a.n_obs + o];
            const double sg = code == 2 ? 1.0 : -1.0;
            lF = -sg * a.V * wn;
        }
        lv[c] = v;
        f[c] = (float)lF;
    }
    return make_float4(f[0], f[1], f[2], a.kappa ? a.kappa[(size_t)b * a.N + i] : 1.0f);
}

// The last step's integrator adjoint (the others follow the bond adjoint of
// the step after them in its kernel).
__global__ void __launch_bounds__(256) k_adj_nodes_st(const __grid_constant__ AdjArgs a, int ls, const double *lu,
                                                      double *lv, float4 *lF4) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= a.N) return;
    const int b = blockIdx.y;
    const size_t n = (size_t)b * a.N + i;
    const double u[3] = {lu[3 * n], lu[3 * n + 1], lu[3 * n + 2]};
    lF4[n] = node_adjoint(a, ls, i, b, u, lv + 3 * n);
}

// The stencil in row order: neighbour offset in the staged tile, xi,
// |xi|, |xi|^2 and 1 / |xi| in FP32.
struct AdjOff {
    int cell;  // bytes
    float x, y, z, L0, L02, iL0, pad;
};
template <int DIM>
struct AdjTab {
    // the last entry pads rows: the node itself at |xi| = dx (no stretch, no terms)
    AdjOff e[2 * Sten<DIM>::kHalf + 1];
};

// Tiles of 8 x TY x TZ nodes (a warp takes 4 rows along y) and a halo of 3;
// TY TZ <= 40, so that the registers of three blocks of at most 320 threads fit
// an SM (64 a thread). Three blocks share it up to about 2,200 cells of records
// (74 KB with the table), two up to the most, 3,072 (96 KB), which thin grids
// reach.
constexpr int kAdjThreads = 320;
constexpr int kMaxCells = 3072;  // 96 KB of records
struct AdjTile {
    int ty, tz, hz;    // nodes; halo layers
    int wy, cells;     // staged rows along y, staged cells
    int ntx, nty, ntz;
};

// The tile that stages the fewest cells over the grid (28k-node beam: 4 x 10
// against 8 x 4 with 256 threads: bond adjoint 430 against 467 us).
AdjTile pick_tile(const pd_grid &g, int hz) {
    AdjTile best = {};
    long long least = 0;
    for (int ty = 4; ty <= 40; ty += 4)
        for (int tz = 1; tz <= 10 && ty * tz <= kAdjThreads / 8; ++tz) {
            AdjTile t = {ty, tz, hz, ty + 2 * kHalo, 0, (g.nx + kSlice - 1) / kSlice, (g.ny + ty - 1) / ty,
                         (g.nz + tz - 1) / tz};
            t.cells = kWx * t.wy * (tz + 2 * hz);
            if (t.cells > kMaxCells) continue;
            const long long staged = (long long)t.nty * t.ntz * t.cells;
            if (!best.ty || staged < least) {
                best = t;
                least = staged;
            }
        }
    return best;
}

struct AdjBond {
    int nz;
    AdjTile t;
    const ulonglong2 *present, *grow, *keep;
    const uint32_t *rows;  // k_adj_rows
    const long long *base;
    const float4 *u4, *lF4;
    float4 *lF4_next;  // of the step before, or nullptr at the run's first step
    int ls;            // this local step
    const float *dprev, *dcur, *d_first;
    float2 *ld;
    double *lu, *lv, *g_s0, *g_k;
    Lay lay;
    long long st_len;
};

// Context of a node's walk over its row.
template <int DIM>
struct AdjNode {
    const AdjArgs &a;
    const AdjBond &g;
    const char *own, *own_l;  // the node's records in the staged tile
    int i, b;
    float4 me, ml;
    float hcV;     // cV / 2
    long long at;  // the node's next growing bond
    float P[5];
};

// One bond. Per bond: y = xi + eta, s = eta.(y + xi) / (|xi| (|y| + |xi|)),
// h = s / |y|, dh/dy = y (1/|xi| - s/|y|) / |y|^2 (|y| from the approximate
// reciprocal square root). special: it grows in the run (damage at this step
// and the next from the trajectory, damage adjoint in double-float), or
// (grows false) keeps a damage other than zero; the damage adjoint of a bond
// that never grows is never used.
struct AdjGrow {
    float dp, dc;  // damage at this step and the next
    float2 ld;     // damage adjoint
};
template <int DIM>
__device__ __forceinline__ void adj_bond(AdjNode<DIM> &n, const AdjOff &o, bool special, bool grows, int e,
                                         const AdjGrow &gr) {
    const float4 nj = *(const float4 *)(n.own + o.cell), lj = *(const float4 *)(n.own_l + o.cell);
    const float xi[3] = {o.x, o.y, o.z};
    const float eta[3] = {nj.x - n.me.x, nj.y - n.me.y, nj.z - n.me.z};
    const float dl[3] = {lj.x - n.ml.x, lj.y - n.ml.y, lj.z - n.ml.z};
    float y[3], y2 = 0.f, num = 0.f, ydl = 0.f;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        y[c] = xi[c] + eta[c];
        y2 = fmaf(y[c], y[c], y2);
        num = fmaf(eta[c], y[c] + xi[c], num);
        ydl = fmaf(y[c], dl[c], ydl);
    }
    const float rL = rsqrt_ap(y2);
    const float L = y2 * rL;
    const float s = num * rcp_ap(fmaf(o.L0, L, o.L02));
    const float h = s * rL;
    const float cijV = n.a.kappa ? n.hcV * (n.ml.w + lj.w) : n.a.cVf;
    const float dhk = rL * rL * (o.iL0 - s * rL);
    if (__builtin_expect(!special, 1)) {  // d = 0: the same roundings as below with om = 1, act = 0
#pragma unroll
        for (int c = 0; c < 3; ++c)
            n.P[c] = __fadd_rn(n.P[c], __fmul_rn(cijV, ydl * dhk * y[c] + h * dl[c]));
        n.P[4] += n.hcV * (-h * ydl);
        return;
    }
    float om, act = 0.f;
    if (grows) {
        const float dp = gr.dp, dc = gr.dc;
        const float2 l0 = gr.ld;
        const bool active = dc > dp;
        const df lamd = df_add(df{l0.x, l0.y}, df{cijV * h * ydl, 0.f});
        float dDds = 0.f, dDds0 = 0.f;
        if (active) law_derivs_f(n.a, s, 0.5f * (n.me.w + nj.w), dDds, dDds0);
        const float lamdf = lamd.hi + lamd.lo;
        om = 1.0f - dc;
        act = active ? lamdf * dDds * rL * o.iL0 : 0.f;
        if (active) n.P[3] += 0.5f * lamdf * dDds0;
        n.g.ld[n.at] = active ? make_float2(0.f, 0.f) : make_float2(lamd.hi, lamd.lo);
        ++n.at;
    } else {
        om = 1.0f - n.g.d_first[(size_t)n.b * n.g.st_len + word_of<DIM>(n.g.lay, n.i, e)];
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) n.P[c] += cijV * om * (ydl * dhk * y[c] + h * dl[c]) - act * y[c];
    n.P[4] += n.hcV * (-om * h * ydl);
}

// The rows of a tile's nodes, lane by lane, padded to the stencil's length:
// four positions over the full stencil to a word, [tile][warp][word][lane] (mesh only, shared by the samples).
template <int DIM>
constexpr int kRowWords = (2 * Sten<DIM>::kHalf + 7) / 8 * 2;
template <int DIM>
__global__ void __launch_bounds__(kAdjThreads) k_adj_rows(int nx, int ny, int nz, const AdjTile t,
                                                          const ulonglong2 *present, uint32_t *rows) {
    const int tile = blockIdx.x, tx = threadIdx.x & 7, ty = threadIdx.x / 8 % t.ty, tz = threadIdx.x / (8 * t.ty);
    const int gx = kSlice * (tile % t.ntx) + tx, gy = t.ty * (tile / t.ntx % t.nty) + ty,
              gz = t.tz * (tile / (t.ntx * t.nty)) + tz;
    if (gx >= nx || gy >= ny || gz >= nz) return;
    const ulonglong2 P = present[gx + (long long)nx * (gy + (long long)ny * gz)];
    uint32_t *o = rows + (((size_t)tile * (blockDim.x >> 5) + (threadIdx.x >> 5)) * kRowWords<DIM>) * 32 + (threadIdx.x & 31);
    uint32_t v = 0u;
    int r = 0;
    for (int h = 0; h < 2; ++h)
        for (unsigned long long w = h ? P.y : P.x; w; w &= w - 1) {
            v |= (uint32_t)(64 * h + __ffsll(w) - 1) << (8 * (r & 3));
            if ((++r & 3) == 0) {
                o[32 * (r / 4 - 1)] = v;
                v = 0u;
            }
        }
    for (; r < 4 * kRowWords<DIM>; ++r) {
        v |= (uint32_t)(2 * Sten<DIM>::kHalf) << (8 * (r & 3));
        if ((r & 3) == 3) {
            o[32 * (r / 4)] = v;
            v = 0u;
        }
    }
}

// Bond adjoint of one step, and the integrator adjoint of the step before it
// (which needs lamu of the node itself only). The lanes of a warp walk their
// own rows in step, whatever bonds they lack, so a node's FP32 sums of 8
// present bonds all end together (walking the full stencil instead, with a
// test per position, the nodes near the faces end theirs at other positions
// than their neighbours, and a warp pays for each).
template <int DIM>
__global__ void __launch_bounds__(kAdjThreads, 3) k_adj_bonds_st(const __grid_constant__ AdjArgs a,
                                                                 const __grid_constant__ AdjBond g,
                                                                 const __grid_constant__ AdjTab<DIM> tab) {
    const AdjTile &T = g.t;
    __shared__ __align__(16) AdjOff s_tab[2 * Sten<DIM>::kHalf + 1];
    extern __shared__ float4 s_rec[];  // (u, s0) of every cell, then (lamF, kappa)
    const int tile = blockIdx.x, b = blockIdx.y;
    const int x0 = kSlice * (tile % T.ntx), y0 = T.ty * (tile / T.ntx % T.nty), z0 = T.tz * (tile / (T.ntx * T.nty));
    const int ny = a.ny, nx = a.nx;
    const float4 *ub = g.u4 + (size_t)b * a.N, *lb4 = g.lF4 + (size_t)b * a.N;
    for (int c = threadIdx.x; c < T.cells; c += blockDim.x) {
        const int r = c / kWx, lz = r / T.wy;
        const int gx = x0 - kHalo + (c - kWx * r), gy = y0 - kHalo + (r - T.wy * lz), gz = z0 - T.hz + lz;
        float4 u = make_float4(0.f, 0.f, 0.f, 0.f), l = u;  // cells outside the grid are never used
        if (gx >= 0 && gx < nx && gy >= 0 && gy < ny && gz >= 0 && gz < g.nz) {
            const int j = gx + nx * (gy + ny * gz);
            u = ub[j];
            l = lb4[j];
        }
        s_rec[c] = u;
        s_rec[T.cells + c] = l;
    }
    for (int e = threadIdx.x; e < 2 * Sten<DIM>::kHalf + 1; e += blockDim.x) s_tab[e] = tab.e[e];
    __syncthreads();
    const int tx = threadIdx.x & 7, ty = threadIdx.x / 8 % T.ty, tz = threadIdx.x / (8 * T.ty);
    const int gx = x0 + tx, gy = y0 + ty, gz = z0 + tz;
    if (gx >= nx || gy >= ny || gz >= g.nz) return;
    const int i = gx + nx * (gy + ny * gz);
    const size_t n = (size_t)b * a.N + i;
    const int own = tx + kHalo + kWx * (ty + kHalo + T.wy * (tz + T.hz));
    float S[5] = {0.f, 0.f, 0.f, 0.f, 0.f}, Cc[5] = {0.f, 0.f, 0.f, 0.f, 0.f};
    AdjNode<DIM> nd{a, g, (const char *)(s_rec + own), (const char *)(s_rec + T.cells + own), i, b, s_rec[own],
                    s_rec[T.cells + own], a.cVf * 0.5f,
                    g.base[n], {0.f, 0.f, 0.f, 0.f, 0.f}};
    const auto fold_all = [&]() {
#pragma unroll
        for (int v = 0; v < 5; ++v) {
            fold(S[v], Cc[v], nd.P[v]);
            nd.P[v] = 0.f;
        }
    };
    const ulonglong2 P = g.present[i];
    const int len = __popcll(P.x) + __popcll(P.y);
    const unsigned lanes = __activemask();  // the tile's nodes inside the grid
    const int W = __reduce_max_sync(lanes, len);
    const uint32_t *rw = g.rows + (((size_t)tile * (blockDim.x >> 5) + (threadIdx.x >> 5)) * kRowWords<DIM>) * 32 +
                         (threadIdx.x & 31);
    const uint32_t *gw = (const uint32_t *)(g.grow + n), *kw = (const uint32_t *)(g.keep + n);
    uint32_t gm = 0u, sm = 0u;
#pragma unroll 1
    for (int p0 = 0; p0 < W; p0 += 8) {
        if ((p0 & 31) == 0) {
            gm = gw[p0 / 32];
            sm = gm | kw[p0 / 32];
        }
        const uint32_t r0 = rw[32 * (p0 / 4)], r1 = rw[32 * (p0 / 4 + 1)];
        if (__any_sync(lanes, sm & 0xffu)) {
            // four at a time: the growing bonds' damage and damage adjoint are
            // requested together
#pragma unroll 1
            for (int h = 0; h < 2; ++h) {
                const uint32_t r = h ? r1 : r0, gh = gm >> (4 * h), sh = sm >> (4 * h);
                AdjGrow gr[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    gr[j] = AdjGrow{0.f, 0.f, make_float2(0.f, 0.f)};
                    if (gh & (1u << j)) {
                        const long long at = nd.at + __popc(gh & ((1u << j) - 1u));
                        gr[j] = AdjGrow{g.dprev[at], g.dcur[at], g.ld[at]};
                    }
                }
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int e = (r >> (8 * j)) & 0xff;
                    adj_bond<DIM>(nd, s_tab[e], sh & (1u << j), gh & (1u << j), e, gr[j]);
                }
            }
        } else {
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const int e = ((j < 4 ? r0 : r1) >> (8 * (j & 3))) & 0xff;
                adj_bond<DIM>(nd, s_tab[e], false, false, e, AdjGrow{});
            }
        }
        gm >>= 8;
        sm >>= 8;
        fold_all();
    }
    double u[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const double carry = a.codes[3 * (size_t)i + c] == 0 ? g.lu[3 * n + c] : 0.0;
        u[c] = carry + ((double)S[c] + (double)Cc[c]);
        g.lu[3 * n + c] = u[c];
    }
    g.g_s0[n] += (double)S[3] + (double)Cc[3];
    if (g.g_k) g.g_k[n] += (double)S[4] + (double)Cc[4];
    if (g.lF4_next) g.lF4_next[n] = node_adjoint(a, g.ls - 1, i, b, u, g.lv + 3 * n);
}

// ---------------------------------------------------------------- host side

struct Bytes {
    char *p = nullptr;
    ~Bytes() { cudaFree(p); }
};

unsigned blocks_of(long long n, int bs) { return (unsigned)((n + bs - 1) / bs); }

// The state's arrays as one checkpoint. Every sample is at step n, whose
// parity selects the records.
struct Checkpoint {
    size_t rec, vdf, dmg, dirty;  // bytes
    size_t bytes() const { return rec + vdf + dmg + dirty; }
    explicit Checkpoint(const pd_state *st) {
        const size_t BN = (size_t)st->B * st->N;
        rec = vdf = 2 * BN * sizeof(float4);
        dmg = (size_t)st->B * st->st_len * sizeof(float);
        dirty = (size_t)st->B * (st->st_len / (st->st_dim == 3 ? Sten<3>::kRounds : Sten<2>::kRounds)) * 4;
        dirty = (dirty + 15) & ~(size_t)15;
    }
    size_t dirty_used(const pd_state *st) const {
        return (size_t)st->B * (st->st_len / (st->st_dim == 3 ? Sten<3>::kRounds : Sten<2>::kRounds)) * 4;
    }
    float *dmg_of(char *p) const { return (float *)(p + rec + vdf); }
    uint32_t *dirty_of(char *p) const { return (uint32_t *)(p + rec + vdf + dmg); }
    int save(const pd_state *st, int n, char *p, cudaStream_t s) const {
        PD_CHECK_CUDA(cudaMemcpyAsync(p, st->rec[n & 1], rec, cudaMemcpyDeviceToDevice, s));
        PD_CHECK_CUDA(cudaMemcpyAsync(p + rec, st->vdf, vdf, cudaMemcpyDeviceToDevice, s));
        PD_CHECK_CUDA(cudaMemcpyAsync(dmg_of(p), st->dmg, dmg, cudaMemcpyDeviceToDevice, s));
        PD_CHECK_CUDA(cudaMemcpyAsync(dirty_of(p), st->st_dirty, dirty_used(st), cudaMemcpyDeviceToDevice, s));
        return PD_OK;
    }
    int restore(pd_state *st, int n, char *p, cudaStream_t s) const {
        PD_TRY(state_set_step(st, n, s));
        for (int q = 0; q < 2; ++q)
            PD_CHECK_CUDA(cudaMemcpyAsync(st->rec[q], p, rec, cudaMemcpyDeviceToDevice, s));
        PD_CHECK_CUDA(cudaMemcpyAsync(st->vdf, p + rec, vdf, cudaMemcpyDeviceToDevice, s));
        PD_CHECK_CUDA(cudaMemcpyAsync(st->dmg, dmg_of(p), dmg, cudaMemcpyDeviceToDevice, s));
        PD_CHECK_CUDA(cudaMemcpyAsync(st->st_dirty, dirty_of(p), dirty_used(st), cudaMemcpyDeviceToDevice, s));
        return stencil_refresh_grec(st, s);
    }
};

// The run bookkeeping of a state, to put back when a call fails after it has
// stepped the state.
struct Bookkeeping {
    int32_t bk_par, rec_off;
    static constexpr int kParts = 9;
    struct Part {
        void *p;
        size_t bytes;
    } part[kParts];
    explicit Bookkeeping(const pd_state *st) : bk_par(st->bk_par), rec_off(st->rec_off) {
        const size_t B = st->B;
        const Part of[kParts] = {{st->step, 8 * B},   {st->done, 8 * B},   {st->pend, 8 * B},
                                 {st->pk2, 16 * B},   {st->ps2, 8 * B},    {st->status, 4 * B},
                                 {st->peak, 8 * B},   {st->peak_step, 4 * B}, {st->ticket, 4 * B}};
        std::copy(of, of + kParts, part);
    }
    static size_t bytes(int B) { return (size_t)kParts * 16 * B; }
    int copy(char *saved, bool back, cudaStream_t s) const {
        for (const Part &q : part) {
            PD_CHECK_CUDA(cudaMemcpyAsync(back ? q.p : saved, back ? saved : q.p, q.bytes, cudaMemcpyDeviceToDevice, s));
            saved += q.bytes;
        }
        return PD_OK;
    }
    int restore(pd_state *st, char *saved, cudaStream_t s) const {
        st->bk_par = bk_par;
        st->rec_off = rec_off;
        return copy(saved, true, s);
    }
};

template <int DIM>
int run(pd_state *st, const AdjArgs &a, int n_steps, int k, const int32_t *steps, double *grad_s0, double *grad_kappa,
        double *R_obs, pd_stream stream) {
    cudaStream_t s = (cudaStream_t)stream;
    const int32_t n0 = steps[0];
    const int B = st->B, nseg = (n_steps + k - 1) / k;
    const long long N = st->N, BN = (long long)B * N;
    PD_REQUIRE(B <= 65535, "at most 65535 samples per state");
    const Checkpoint ck(st);
    const AdjTile T = pick_tile(st->g, Sten<DIM>::kHaloZ);
    const unsigned tiles = (unsigned)(T.ntx * T.nty * T.ntz), threads = 8u * T.ty * T.tz;
    // one allocation: checkpoints and the final state, FP32 node records of a
    // segment, (lamF, kappa) of two steps, lamu, lamv, reactions, masks, list starts and the run bookkeeping
    size_t off = 0;
    const auto part = [&](size_t bytes) {
        const size_t at = off;
        off += (bytes + 255) & ~(size_t)255;
        return at;
    };
    const size_t o_ck = part((size_t)(nseg + 1) * ck.bytes()), o_u4 = part((size_t)k * BN * sizeof(float4)),
                 o_lF = part(2 * BN * sizeof(float4)), o_lu = part(3 * BN * sizeof(double)),
                 o_lv = part(3 * BN * sizeof(double)), o_r = part((size_t)B * k * sizeof(double)),
                 o_rows = part((size_t)tiles * (threads / 32) * kRowWords<DIM> * 32 * sizeof(uint32_t)),
                 o_pm = part(N * sizeof(ulonglong2)), o_gm = part(BN * sizeof(ulonglong2)),
                 o_km = part(BN * sizeof(ulonglong2)), o_base = part((BN + 1) * sizeof(long long)),
                 o_bk = part(Bookkeeping::bytes(B));
    Bytes mem;
    PD_TRY(dalloc(&mem.p, off));
    const auto ck_at = [&](int g) { return mem.p + o_ck + (size_t)g * ck.bytes(); };
    float4 *u4 = (float4 *)(mem.p + o_u4), *lF4 = (float4 *)(mem.p + o_lF);
    double *lu = (double *)(mem.p + o_lu), *lv = (double *)(mem.p + o_lv), *rbuf = (double *)(mem.p + o_r);
    ulonglong2 *pm = (ulonglong2 *)(mem.p + o_pm), *gm = (ulonglong2 *)(mem.p + o_gm), *km = (ulonglong2 *)(mem.p + o_km);
    long long *base = (long long *)(mem.p + o_base);
    uint32_t *rows = (uint32_t *)(mem.p + o_rows);

    const Bookkeeping bk(st);
    PD_TRY(bk.copy(mem.p + o_bk, false, s));

    // forward with checkpoints (the step set first clears run bookkeeping, e.g. done flags)
    if (std::any_of(steps, steps + B, [&](int32_t n) { return (n ^ n0) & 1; })) {
        k_adj_align<<<dim3(blocks_of(N, 256), B), 256, 0, s>>>(N, BN, st->step + st->bk_par * B, n0, (float4 *)st->rec[0],
                                                              (float4 *)st->rec[1]);
        PD_CHECK_LAUNCH();
        PD_TRY(stencil_refresh_grec(st, s));
    }
    PD_TRY(state_set_step(st, n0, s));
    for (int g = 0; g < nseg; ++g) {
        const int start = g * k, len = std::min(k, n_steps - start);
        PD_TRY(ck.save(st, n0 + start, ck_at(g), s));
        PD_TRY(pd_step(st, len, rbuf, stream));
        if (R_obs && a.n_obs) PD_TRY(adjoint_gather_obs(B, len, start, a.n_obs, a.obs, rbuf, R_obs, s));
    }
    PD_TRY(ck.save(st, n0 + n_steps, ck_at(nseg), s));

    // the growing bonds
    Lay y;
    y.nx = st->g.nx;
    y.ny = st->g.ny;
    y.nz = st->g.nz;
    y.BY = st->by;
    y.BZ = st->bz;
    y.nbx = st->nbx;
    y.nby = st->nby;
    y.wpb = st->st_wpb;
    y.n_rp = st->n_bricks * st->st_wpb;
    y.N = N;
    k_adj_masks<DIM><<<dim3(blocks_of(y.n_rp, 8), B), 256, 0, s>>>(
        y, (const float4 *)st->st_tmpl, (const float4 *)ck.dmg_of(ck_at(0)), (const float4 *)ck.dmg_of(ck_at(nseg)),
        ck.dirty_of(ck_at(nseg)), st->st_q, pm, gm, km, base);
    PD_CHECK_LAUNCH();
    k_adj_rows<DIM><<<tiles, threads, 0, s>>>(st->g.nx, st->g.ny, st->g.nz, T, pm, rows);
    PD_CHECK_LAUNCH();
    const long long nblk = (BN + 1023) / 1024;
    k_scan64_blocks<<<(unsigned)nblk, 1024, 0, s>>>(base, BN);
    PD_CHECK_LAUNCH();
    k_scan64_ends<<<1, 1024, 0, s>>>(base, BN, nblk);
    PD_CHECK_LAUNCH();
    if (nblk > 1) {
        k_scan64_add<<<(unsigned)(nblk - 1), 1024, 0, s>>>(base, BN);
        PD_CHECK_LAUNCH();
    }
    long long n_grow = 0;
    PD_CHECK_CUDA(cudaMemcpyAsync(&n_grow, base + BN, sizeof(n_grow), cudaMemcpyDeviceToHost, s));
    PD_CHECK_CUDA(cudaStreamSynchronize(s));
    const size_t ng = (size_t)std::max(n_grow, 1ll);
    const bool wide = st->st_len > (1ll << 32);  // a sample's damage words
    off = 0;
    const size_t o_tr = part((size_t)(k + 1) * ng * sizeof(float)), o_ld = part(ng * sizeof(float2)),
                 o_words = part(ng * (wide ? sizeof(uint64_t) : sizeof(uint32_t)));
    Bytes gmem;
    const int grc = dalloc(&gmem.p, off);
    if (grc != PD_OK) {  // the state as the call found it
        PD_TRY(ck.restore(st, n0, ck_at(0), s));
        PD_TRY(bk.restore(st, mem.p + o_bk, s));
        PD_CHECK_CUDA(cudaStreamSynchronize(s));
        return grc;
    }
    float *tr_d = (float *)(gmem.p + o_tr);
    float2 *ld = (float2 *)(gmem.p + o_ld);
    uint32_t *words = (uint32_t *)(gmem.p + o_words);
    uint64_t *words64 = (uint64_t *)(gmem.p + o_words);
    if (wide)
        k_adj_list<DIM><<<blocks_of(BN, 256), 256, 0, s>>>(y, B, pm, gm, base, words64);
    else
        k_adj_list<DIM><<<blocks_of(BN, 256), 256, 0, s>>>(y, B, pm, gm, base, words);
    PD_CHECK_LAUNCH();
    PD_CHECK_CUDA(cudaMemsetAsync(ld, 0, ng * sizeof(float2), s));
    PD_CHECK_CUDA(cudaMemsetAsync(lu, 0, 3 * BN * sizeof(double), s));
    PD_CHECK_CUDA(cudaMemsetAsync(lv, 0, 3 * BN * sizeof(double), s));
    PD_CHECK_CUDA(cudaMemsetAsync(grad_s0, 0, BN * sizeof(double), s));
    if (grad_kappa) PD_CHECK_CUDA(cudaMemsetAsync(grad_kappa, 0, BN * sizeof(double), s));

    AdjTab<DIM> tab = {};
    constexpr int H = Sten<DIM>::kHalf;
    for (int m = 0; m < H; ++m)
        for (int t = 0; t < 2; ++t) {
            const I3 o = half_off<DIM>(m);
            const int sg = t ? -1 : 1, q2 = o.x * o.x + o.y * o.y + o.z * o.z;
            AdjOff &e = tab.e[row_pos<DIM>(m, t)];
            e.cell = sg * (o.x + kWx * (o.y + T.wy * o.z)) * (int)sizeof(float4);
            e.x = (float)(sg * o.x) * a.dxf;
            e.y = (float)(sg * o.y) * a.dxf;
            e.z = (float)(sg * o.z) * a.dxf;
            e.L0 = a.L0q[q2];
            e.L02 = e.L0 * e.L0;
            e.iL0 = a.iL0q[q2];
            e.pad = 0.f;
        }
    {
        AdjOff &e = tab.e[2 * H];
        e.x = a.dxf;
        e.L0 = a.L0q[1];
        e.L02 = e.L0 * e.L0;
        e.iL0 = a.iL0q[1];
    }
    AdjBond bo = {};
    bo.nz = st->g.nz;
    bo.t = T;
    bo.rows = rows;
    bo.present = pm;
    bo.grow = gm;
    bo.keep = km;
    bo.base = base;
    bo.d_first = ck.dmg_of(ck_at(0));
    bo.ld = ld;
    bo.lu = lu;
    bo.lv = lv;
    bo.g_s0 = grad_s0;
    bo.g_k = grad_kappa;
    bo.lay = y;
    bo.st_len = st->st_len;
    const size_t smem = 2 * sizeof(float4) * T.cells;
    PD_CHECK_CUDA(cudaFuncSetAttribute(k_adj_bonds_st<DIM>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(2 * sizeof(float4) * kMaxCells)));
    const dim3 snap_grid((unsigned)std::max(1, std::min(64, (int)blocks_of(N, 256))), (unsigned)B);
    const auto snap = [&](const float4 *rec, float4 *dst, float *d) -> int {
        if (wide)
            k_adj_snap<<<snap_grid, 256, 0, s>>>(N, BN, base, words64, (const float *)st->dmg, st->st_len, d, rec, dst);
        else
            k_adj_snap<<<snap_grid, 256, 0, s>>>(N, BN, base, words, (const float *)st->dmg, st->st_len, d, rec, dst);
        PD_CHECK_LAUNCH();
        return PD_OK;
    };
    for (int g = nseg - 1; g >= 0; --g) {
        const int start = g * k, len = std::min(k, n_steps - start);
        PD_TRY(ck.restore(st, n0 + start, ck_at(g), s));
        for (int m = 0; m < len; ++m) {
            PD_TRY(snap((const float4 *)st->rec[(n0 + start + m) & 1], u4 + (size_t)m * BN, tr_d + (size_t)m * ng));
            PD_TRY(pd_step(st, 1, nullptr, stream));
        }
        PD_TRY(snap(nullptr, nullptr, tr_d + (size_t)len * ng));
        if (g == nseg - 1) {
            k_adj_nodes_st<<<dim3(blocks_of(N, 256), B), 256, 0, s>>>(a, n_steps - 1, lu, lv, lF4);
            PD_CHECK_LAUNCH();
        }
        for (int m = len - 1; m >= 0; --m) {
            const int ls = start + m, cur = (n_steps - 1 - ls) & 1;
            bo.u4 = u4 + (size_t)m * BN;
            bo.lF4 = lF4 + (size_t)cur * BN;
            bo.lF4_next = ls > 0 ? lF4 + (size_t)(1 - cur) * BN : nullptr;
            bo.ls = ls;
            bo.dprev = tr_d + (size_t)m * ng;
            bo.dcur = tr_d + (size_t)(m + 1) * ng;
            k_adj_bonds_st<DIM><<<dim3(tiles, B), threads, smem, s>>>(a, bo, tab);
            PD_CHECK_LAUNCH();
        }
    }
    // leave the state where the forward run left it
    PD_TRY(ck.restore(st, n0 + n_steps, ck_at(nseg), s));
    if (cudaStreamSynchronize(s) != cudaSuccess) {
        set_error("adjoint failed: %s", cudaGetErrorString(cudaGetLastError()));
        return PD_ERR_CUDA;
    }
    return PD_OK;
}

}  // namespace

int adjoint_stencil(pd_state *st, const AdjArgs &a, int n_steps, int k, const int32_t *steps, double *grad_s0,
                    double *grad_kappa, double *R_obs, pd_stream stream) {
    return st->st_dim == 3 ? run<3>(st, a, n_steps, k, steps, grad_s0, grad_kappa, R_obs, stream)
                           : run<2>(st, a, n_steps, k, steps, grad_s0, grad_kappa, R_obs, stream);
}

}  // namespace pdi
