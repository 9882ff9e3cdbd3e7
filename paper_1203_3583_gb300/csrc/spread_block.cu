// Atomic-free spread of monotone maps by block items merged in four colours:
// kernel widths 8 to 16, and the deterministic plans of every width.
//
// A block item is a rectangle of source samples.  Its warps walk down source
// columns; each lane keeps the taps of its column in a register window of W
// rows that slides down the fine grid with the samples (spread.cuh), and adds
// a row that leaves the window to a tile of shared memory private to its warp.
// At the end the block adds its warps' tiles to the fine grid.
//
//  * Width.  W x W complex cells do not fit a lane's registers above W = 7, so
//    S lanes (2 up to width 12, else 4) share a source column: lane group `sub`
//    holds the tap columns [sub WS, sub WS + WS), WS = W / S rounded up.  The
//    groups of a warp have tiles of their own, so that groups never meet.
//  * No atomics within a warp.  All rows that leave the windows in a step do so
//    in warp-uniform phases, window row by row and column by column, with a
//    warp barrier between phases; in a phase two lanes of a group meet in a cell
//    only if their first taps are the same.  Where neighbouring samples can be
//    less than a cell apart (DUP) such lanes' rows are first added up over the
//    lanes, in lane order, and written by the first of them.
//  * No atomics between blocks.  Blocks are launched in four colours (parity
//    of their column and row of blocks), and the plan makes blocks large enough
//    that blocks of one colour never touch the same cell: a block adds its sums
//    to the grid with plain loads and stores, and each cell receives its
//    contributions in the order of the colours.  The grid's band must be zero
//    before (the row pass leaves it so).
//
// Results are therefore bit-identical from run to run.
//
// What bounds it: a warp's chain of latencies per source row (ring, position,
// phases), at 8 warps per SM (230 registers at W = 12: 144 are the window).
// Measured, whole transforms, against the conflict-free tiles and, for maps
// denser than 64 samples per kernel width and widths above 14, the shared-memory
// float atomics that these maps took before (us):
//   2048^2, 1.04 cells per sample   w8 506 -> 218, w12 1407 -> 356, w16 3433 -> 695
//   600^2 onto 256^2 (0.4 cells)    w7 487 -> 109, w8 1221 -> 93, w12 3774 -> 139
//   1300 x 1258 onto 64^2 (0.03)    w7 211500 -> 1789, w12 606400 -> 5317
// Maps whose samples lie cells apart keep the tiles (kSparse in plan.cu).
// Sharing a column between 4 lanes at W = 12 (half the registers, twice the
// steps) took 1.45 times as long.
#include <algorithm>
#include <climits>
#include <cmath>
#include <vector>

#include "fft.cuh"
#include "spread.cuh"

namespace asfd {

namespace {

constexpr int kBlkMaxWarps = 8;
constexpr size_t kBlkMaxSmem = 200 * 1024;

__host__ __device__ constexpr int blk_split(int w) { return spread_split(w); }
__host__ __device__ constexpr int blk_cols(int w) { return (w + blk_split(w) - 1) / blk_split(w); }
// bytes of the input ring of a warp: u1, q and the row's table entries of
// kDenseRing rows
__host__ __device__ constexpr int blk_ring(int w) { return kDenseRing * ((32 / blk_split(w)) * 12 + 32); }

struct BlkArgs {
    SpreadArgs s;
    const int* xbox;  // [warp columns][2]: first tap columns' range [lo, hi) and its taps
    const int* ybox;  // [block rows][2]
    int chunks;       // column chunks (32 / S columns each) that a warp takes in turn
    int rows;         // source rows of a block
    int ncols;        // warp columns in all
    int nbx, nby;     // block columns and rows in all
    int cx, cy;       // this launch's colour
    int tw, th;       // tile of a lane group (cells)
};

// Weights of W taps in y, then WS taps (from tap0) in x, two at a time: pair k
// of the W + WS (the last may be alone).
template <int W, int WS>
__device__ __forceinline__ void blk_weight_pair(const SpreadArgs& a, float neg_c2, float zy, float zx,
                                                int k, float (&e)[W + WS + 1])
{
    const int k0 = 2 * k, k1 = 2 * k + 1;
    const float z0 = k0 < W ? zy + (float)k0 : zx + (float)(k0 - W);
    const float z1 = k1 < W ? zy + (float)k1 : zx + (float)(k1 - W);
    const float2 v = es_weight2_fast(make_float2(z0, z1), neg_c2, a.beta_log2e);
    e[k0] = v.x;
    e[k1] = v.y;
}

// Adds a sample to a window: fresh (every slot is overwritten), or with its
// first tap row d = 0, 1 or 2 rows below the window's (whose d top rows have
// left it: the rest moves up inside the multiply-adds).
template <int W, int WS>
__device__ __forceinline__ void blk_accumulate(float2 (&acc)[W][WS], bool fresh, int d, float2 c,
                                               const float (&wy)[W], const float (&wx)[WS])
{
    if (fresh) {
#pragma unroll
        for (int b = 0; b < W; ++b) {
            const float2 cb = mul2(c, wy[b]);
#pragma unroll
            for (int i = 0; i < WS; ++i) acc[b][i] = mul2(cb, wx[i]);
        }
    } else if (d == 0) {
#pragma unroll
        for (int b = 0; b < W; ++b) {
            const float2 cb = mul2(c, wy[b]);
#pragma unroll
            for (int i = 0; i < WS; ++i) acc[b][i] = fma2(cb, wx[i], acc[b][i]);
        }
    } else if (d == 1) {
#pragma unroll
        for (int b = 0; b < W; ++b) {
            const float2 cb = mul2(c, wy[b]);
#pragma unroll
            for (int i = 0; i < WS; ++i)
                acc[b][i] = (b + 1 < W) ? fma2(cb, wx[i], acc[b + 1][i]) : mul2(cb, wx[i]);
        }
    } else {
#pragma unroll
        for (int b = 0; b < W; ++b) {
            const float2 cb = mul2(c, wy[b]);
#pragma unroll
            for (int i = 0; i < WS; ++i)
                acc[b][i] = (b + 2 < W) ? fma2(cb, wx[i], acc[b + 2][i]) : mul2(cb, wx[i]);
        }
    }
}

template <int W, bool DUP>
__global__ void __launch_bounds__(32 * kBlkMaxWarps) spread_block_kernel(BlkArgs ba)
{
    constexpr int S = blk_split(W), WS = blk_cols(W), HC = 32 / S;
    constexpr unsigned full = 0xffffffffu;
    // prefactors with the accurate sine and cosine: the widths asked for where the
    // last digits matter, and the maps of many samples per kernel width
    constexpr bool ACCURATE = DUP || W > kMaxRingWidth;
    extern __shared__ float4 blk_smem[];
    chain_next();
    chain_wait();
    const SpreadArgs& a = ba.s;
    const int warps = blockDim.x / 32, wid = threadIdx.x / 32, lane = threadIdx.x % 32;
    const int sub = lane / HC, slot = lane % HC;
    const int tw = ba.tw, th = ba.th, tcells = tw * th;
    char* ring = reinterpret_cast<char*>(blk_smem) + wid * blk_ring(W);
    float2* tiles = reinterpret_cast<float2*>(reinterpret_cast<char*>(blk_smem) + warps * blk_ring(W));
    float2* tile = tiles + (size_t)(wid * S + sub) * tcells;
    const int bx = 2 * blockIdx.x + ba.cx, by = 2 * blockIdx.y + ba.cy;
    const int wc = bx * warps + wid;  // warp column
    const int ny0 = by * ba.rows, nyl = min(ny0 + ba.rows, a.n1y) - 1;
    const int ylo = ba.ybox[2 * by];

    for (int i = threadIdx.x; i < warps * S * tcells; i += blockDim.x) tiles[i] = make_float2(0.f, 0.f);
    __syncthreads();

    const float neg_c2 = -a.two_over_w * a.two_over_w;
    float2* ring_u = reinterpret_cast<float2*>(ring);
    float* ring_q = reinterpret_cast<float*>(ring_u + kDenseRing * HC);
    char* ring_t = reinterpret_cast<char*>(ring_q + kDenseRing * HC);
    const int xlo = wc < ba.ncols ? ba.xbox[2 * wc] : 0;
    for (int ch = 0; ch < ba.chunks; ++ch) {
        const int nx0 = (wc * ba.chunks + ch) * HC;
        if (wc >= ba.ncols || nx0 >= a.n1x) break;  // warp-uniform
        // lanes past the last column follow the last one without flushing
        const bool lane_on = nx0 + slot < a.n1x;
        const int nx = lane_on ? nx0 + slot : a.n1x - 1;
        const AxisEntry ex = a.ax[nx];
        const AxisPos px = a.px[nx];
        float2 acc[W][WS];
        int X0 = 0, R0 = 0;
        bool live = false;
        // window rows b < nflush go to the tile, in phases over the window's
        // columns; where first taps of a row can coincide (DUP) row by row
        auto flush = [&](int nflush, int nb) {
            const int c0 = X0 - xlo, r0 = R0 - ylo;
            float2* p = tile + r0 * tw + c0;
            if constexpr (!DUP) {
#pragma unroll
                for (int i = 0; i < WS; ++i) {
                    const bool in = lane_on && (unsigned)(c0 + i) < (unsigned)tw;
#pragma unroll
                    for (int b = 0; b < W; ++b) {
                        if (b >= nb) break;  // warp-uniform
                        if (in && b < nflush && (unsigned)(r0 + b) < (unsigned)th)
                            p[b * tw + i] = cadd(p[b * tw + i], acc[b][i]);
                    }
                    __syncwarp(full);
                }
            } else {
                // lanes of this group with the same first tap
                const bool any = lane_on && nflush > 0;
                unsigned grp = __match_any_sync(full, any ? ((unsigned)R0 << 16 | (unsigned)X0) : ~(unsigned)lane);
                grp &= (HC == 32 ? full : ((1u << (HC & 31)) - 1u)) << (sub * HC);
#pragma unroll
                for (int b = 0; b < W; ++b) {
                    if (b >= nb) break;  // warp-uniform
                    bool on = lane_on && b < nflush && (unsigned)(r0 + b) < (unsigned)th;
                    const unsigned mem = grp & __ballot_sync(full, on);
                    const int most = __reduce_max_sync(full, on ? __popc(mem) : 0);
                    const int first = on ? __ffs(mem) - 1 : lane;
                    unsigned rest = on ? mem & (mem - 1) : 0;
                    for (int k = 1; k < most; ++k) {
                        const int src = rest ? __ffs(rest) - 1 : lane;
                        const bool take = on && first == lane && rest;
                        rest &= rest - 1;
#pragma unroll
                        for (int i = 0; i < WS; ++i) {
                            const float vx = __shfl_sync(full, acc[b][i].x, src);
                            const float vy = __shfl_sync(full, acc[b][i].y, src);
                            if (take) acc[b][i] = cadd(acc[b][i], make_float2(vx, vy));
                        }
                    }
                    on = on && first == lane;
#pragma unroll
                    for (int i = 0; i < WS; ++i) {
                        if (on && (unsigned)(c0 + i) < (unsigned)tw)
                            p[b * tw + i] = cadd(p[b * tw + i], acc[b][i]);
                        __syncwarp(full);
                    }
                }
            }
        };
        // u1 and q of the chunk's columns and the row's y table entries, a
        // kDenseAhead-row cp.async ring as in the default spread
        auto issue_row = [&](int r) {
            if (r <= nyl) {
                const size_t n = (size_t)r * a.n1x + nx;
                const int sl = (r - ny0) & (kDenseRing - 1);
                if (S == 1 || sub == 0) {
                    const unsigned du = (unsigned)__cvta_generic_to_shared(ring_u + sl * HC + slot);
                    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(du), "l"(a.u1 + n));
                }
                if (S == 1 || sub == 1) {
                    const unsigned dq = (unsigned)__cvta_generic_to_shared(ring_q + sl * HC + slot);
                    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dq), "l"(a.q + n));
                }
                if (lane == 0) {
                    const unsigned dt = (unsigned)__cvta_generic_to_shared(ring_t + sl * 32);
                    asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(dt), "l"(a.ay + r));
                    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(dt + 16), "l"(a.py + r));
                }
            }
            asm volatile("cp.async.commit_group;");
        };
        __syncwarp(full);  // every lane is done with the previous chunk's ring
#pragma unroll
        for (int r = 0; r < kDenseAhead; ++r) issue_row(ny0 + r);
        for (int ny = ny0; ny <= nyl; ++ny) {
            asm volatile("cp.async.wait_group %0;" ::"n"(kDenseAhead - 1));
            __syncwarp(full);
            const int sl = (ny - ny0) & (kDenseRing - 1);
            const AxisEntry ey = *reinterpret_cast<const AxisEntry*>(ring_t + sl * 32);
            const AxisPos py = *reinterpret_cast<const AxisPos*>(ring_t + sl * 32 + 16);
            const float q = ring_q[sl * HC + slot];
            const float2 u = ring_u[sl * HC + slot];
            issue_row(ny + kDenseAhead);
            int l0x, l0y;
            float dx, dy;
            sample_pos(ex, ey, px, py, q, a.half_w, l0x, l0y, dx, dy);
            const int d = l0y - R0;
            const bool restart = live && (l0x != X0 || d < 0 || d > 2);
            const int nflush = restart ? W : (live ? d : 0);
            const int nb = __reduce_max_sync(full, lane_on ? nflush : 0);
            constexpr int PAIRS = (W + WS + 1) / 2;
            const float zy = dy - a.half_w, zx = dx - a.half_w + (float)(sub * WS);
            float e[W + WS + 1];
            if (!DUP && nb == 1) {
                // the usual step: the weights' arithmetic fills the phases' waits
                const int c0 = X0 - xlo, r0 = R0 - ylo;
                float2* p = tile + r0 * tw + c0;
                const bool on = lane_on && nflush == 1 && (unsigned)r0 < (unsigned)th;
#pragma unroll
                for (int i = 0; i < WS; ++i) {
                    const bool in = on && (unsigned)(c0 + i) < (unsigned)tw;
                    float2 v = make_float2(0.f, 0.f);
                    if (in) v = p[i];
#pragma unroll
                    for (int k = i * PAIRS / WS; k < (i + 1) * PAIRS / WS; ++k)
                        blk_weight_pair<W, WS>(a, neg_c2, zy, zx, k, e);
                    if (in) p[i] = cadd(v, acc[0][i]);
                    __syncwarp(full);
                }
            } else {
                if (nb > 0) flush(nflush, nb);
#pragma unroll
                for (int k = 0; k < PAIRS; ++k) blk_weight_pair<W, WS>(a, neg_c2, zy, zx, k, e);
            }
            float wx[WS], wy[W];
#pragma unroll
            for (int b = 0; b < W; ++b) wy[b] = e[b];
            // (taps beyond W, in the last group where S does not divide W)
#pragma unroll
            for (int i = 0; i < WS; ++i) wx[i] = (S * WS > W && sub * WS + i >= W) ? 0.f : e[W + i];
            const bool fresh = !live || restart;
            if (fresh) {
                X0 = l0x;
                live = true;
            }
            R0 = l0y;
            const float2 c = ACCURATE ? sample_value(u, ex, ey, q, a.inc_d)
                                      : sample_value_fast(u, ex, ey, q, a.inc_d);
            blk_accumulate<W, WS>(acc, fresh, d, c, wy, wx);
        }
        flush(live ? W : 0, W);
        asm volatile("cp.async.wait_group 0;");
    }
    __syncthreads();

    // the block's footprint: a thread per column, over a share of the rows; the
    // tiles of the lane groups that cover the column in a fixed order
    const int wc0 = bx * warps, wcn = min(warps, ba.ncols - wc0);
    const int gx0 = ba.xbox[2 * wc0], gx1 = ba.xbox[2 * (wc0 + wcn - 1) + 1];
    const int gy0 = ylo, gy1 = ba.ybox[2 * by + 1];
    const int band_x1 = (a.band_tx0 + a.band_ntx) * kTileX;
    const int xb = max(gx0, a.band_tx0 * kTileX), xe = min(gx1, band_x1);
    // (gy0 + th: the boxes of a replayed launch may be those of a later map)
    const int yb = max(gy0, 0), ye = min(min(gy1, a.nfy), gy0 + th);
    const int across = max(1, (xe - xb + 31) / 32) * 32;          // threads along x
    const int parts = max(1, (int)blockDim.x / across);           // shares of the rows
    const int part = (int)threadIdx.x / across;
    if (part >= parts && across <= (int)blockDim.x) return;
    const int x0 = across <= (int)blockDim.x ? (int)threadIdx.x % across : (int)threadIdx.x;
    const int ypart = across <= (int)blockDim.x ? part : 0;
    for (int x = xb + x0; x < xe; x += min(across, (int)blockDim.x)) {
        // (warp, group) tiles whose columns [lo, lo + tw) hold x
        unsigned cover = 0;
        for (int t = 0; t < wcn * S; ++t) {
            const int c = x - ba.xbox[2 * (wc0 + t / S)] - (t % S) * WS;
            if ((unsigned)c < (unsigned)tw) cover |= 1u << t;
        }
        constexpr int R = 4;  // rows whose loads are in flight together
        for (int y = yb + ypart; y < ye; y += R * parts) {
            float2 s[R];
#pragma unroll
            for (int k = 0; k < R; ++k)
                if (y + k * parts < ye) s[k] = a.grid[(size_t)(y + k * parts) * a.nfx + x];
            for (unsigned m = cover; m; m &= m - 1) {
                const int t = __ffs(m) - 1;
                const int c = x - ba.xbox[2 * (wc0 + t / S)] - (t % S) * WS;
                const float2* v = tiles + (size_t)t * tcells + (y - gy0) * tw + c;
#pragma unroll
                for (int k = 0; k < R; ++k)
                    if (y + k * parts < ye) s[k] = cadd(s[k], v[k * parts * tw]);
            }
#pragma unroll
            for (int k = 0; k < R; ++k)
                if (y + k * parts < ye) a.grid[(size_t)(y + k * parts) * a.nfx + x] = s[k];
        }
    }
}

// Folding or wrapping maps at widths above kMaxWindowWidth: the windows of the
// block items (S lanes share a source column), flushed to wrapped cells of the
// fine grid with float2 atomic adds.  Warp item `it` takes 32 / S columns over
// dense_rows rows.  Any map is handled: a sample that does not continue its
// lane's window flushes it.  (Shared-memory tiles with float atomics, a
// compare-and-swap loop each and one block per 64 x 64 cells, took 1093 us for a
// wrapping 1024^2 onto 512^2 at w12, now 59; 205 ms for 1300 x 1258 onto 64^2, now
// 0.09; 1178 us for a folding 1024^2, now 304.)
template <int W>
__global__ void __launch_bounds__(32 * kDenseWarps) spread_fold_kernel(SpreadArgs a)
{
    constexpr int S = blk_split(W), WS = blk_cols(W), HC = 32 / S, PAIRS = (W + WS + 1) / 2;
    chain_next();
    chain_wait();
    const int it = blockIdx.x * kDenseWarps + threadIdx.x / 32, lane = threadIdx.x % 32;
    const int sub = lane / HC, slot = lane % HC;
    const int ncb = (a.n1x + HC - 1) / HC;
    const int nx = (it % ncb) * HC + slot;
    const int ny0 = (it / ncb) * a.dense_rows;
    const int nyl = min(ny0 + a.dense_rows, a.n1y) - 1;
    if (it >= a.dense_items || nx >= a.n1x || ny0 > nyl) return;
    const int mx = a.nfx - 1, my = a.nfy - 1;
    const float neg_c2 = -a.two_over_w * a.two_over_w;
    const AxisEntry ex = a.ax[nx];
    const AxisPos px = a.px[nx];
    float2 acc[W][WS];
    int X0 = 0, R0 = 0;
    bool live = false;
    auto flush = [&](int n) {
#pragma unroll
        for (int b = 0; b < W; ++b) {
            if (b >= n) break;
            float2* row = a.grid + (size_t)((R0 + b) & my) * a.nfx;
#pragma unroll
            for (int i = 0; i < WS; ++i)
                if (S * WS == W || sub * WS + i < W)
                    atomicAdd(row + ((X0 + sub * WS + i) & mx), acc[b][i]);
        }
    };
    size_t n = (size_t)ny0 * a.n1x + nx;
    float qn = __ldg(&a.q[n]);
    float2 un = a.u1[n];
    for (int ny = ny0; ny <= nyl; ++ny) {
        const float q = qn;
        const float2 u = un;
        n += a.n1x;
        if (ny < nyl) {
            qn = __ldg(&a.q[n]);
            un = a.u1[n];
        }
        const AxisEntry ey = a.ay[ny];
        int l0x, l0y;
        float dx, dy;
        sample_pos(ex, ey, px, a.py[ny], q, a.half_w, l0x, l0y, dx, dy);
        const int d = l0y - R0;
        const bool fresh = !live || l0x != X0 || d < 0 || d > 2;
        if (live) flush(fresh ? W : d);
        X0 = l0x;
        R0 = l0y;
        live = true;
        const float2 c = sample_value(u, ex, ey, q, a.inc_d);
        float e[W + WS + 1];
        const float zy = dy - a.half_w, zx = dx - a.half_w + (float)(sub * WS);
#pragma unroll
        for (int k = 0; k < PAIRS; ++k) blk_weight_pair<W, WS>(a, neg_c2, zy, zx, k, e);
        float wx[WS], wy[W];
#pragma unroll
        for (int b = 0; b < W; ++b) wy[b] = e[b];
#pragma unroll
        for (int i = 0; i < WS; ++i) wx[i] = e[W + i];
        blk_accumulate<W, WS>(acc, fresh, d, c, wy, wx);
    }
    flush(W);
}

using BlkKernel = void (*)(BlkArgs);

template <bool DUP>
BlkKernel blk_kernel(int w)
{
    switch (w) {
#define ASFD_BK(W) case W: return spread_block_kernel<W, DUP>;
        ASFD_BK(2) ASFD_BK(3) ASFD_BK(4) ASFD_BK(5) ASFD_BK(6) ASFD_BK(7) ASFD_BK(8) ASFD_BK(9)
        ASFD_BK(10) ASFD_BK(11) ASFD_BK(12) ASFD_BK(13) ASFD_BK(14) ASFD_BK(15) ASFD_BK(16)
#undef ASFD_BK
        default: return nullptr;
    }
}

}  // namespace

// Chooses the block items of a monotone map without wrap from the ranges of
// its columns' x and rows' y storage coordinates (cr, rr: [lo, hi] pairs), and
// uploads their boxes; P->blk stays false where no shape fits.
asfd_status plan_build_block(asfd_plan_s* P, const std::vector<double>& cr,
                             const std::vector<double>& rr, cudaStream_t st)
{
    const asfd_params& p = P->prm;
    P->blk = false;
    const int w = P->w, S = blk_split(w), WS = blk_cols(w), HC = 32 / S;
    // first taps of coordinate g: ceil(g - w/2), with a margin for FP32
    const auto first = [&](double g) { return (int)std::floor(g - 0.5 * w - 0.01); };
    const auto last = [&](double g) { return (int)std::ceil(g - 0.5 * w + 0.01) + w; };
    // ranges of groups of `step` consecutive entries
    const auto boxes = [&](const std::vector<double>& r, int n, int step) {
        std::vector<int> b;
        for (int i = 0; i < n; i += step) {
            int lo = INT_MAX, hi = INT_MIN;
            for (int k = i; k < std::min(n, i + step); ++k) {
                lo = std::min(lo, first(r[2 * k]));
                hi = std::max(hi, last(r[2 * k + 1]));
            }
            b.push_back(lo);
            b.push_back(hi);
        }
        return b;
    };
    // groups two apart must not share a cell, and boxes must move forward
    const auto separate = [](const std::vector<int>& b, size_t per) {
        const size_t n = b.size() / 2;
        std::vector<int> lo, hi;
        for (size_t i = 0; i < n; i += per) {
            lo.push_back(b[2 * i]);
            hi.push_back(b[2 * i + 1]);
            for (size_t k = i; k < std::min(n, i + per); ++k) {
                lo.back() = std::min(lo.back(), b[2 * k]);
                hi.back() = std::max(hi.back(), b[2 * k + 1]);
            }
        }
        for (size_t i = 0; i + 1 < lo.size(); ++i) {
            if (lo[i + 1] < lo[i] || hi[i + 1] < hi[i]) return false;
            if (i + 2 < lo.size() && hi[i] > lo[i + 2]) return false;
        }
        return true;
    };
    const auto widest = [](const std::vector<int>& b) {
        int m = 0;
        for (size_t i = 0; i < b.size(); i += 2) m = std::max(m, b[i + 1] - b[i]);
        return m;
    };
    // (beyond 64 samples per kernel width: see ACCURATE)
    bool dup = P->min_step_x < 1.0 + 1e-3 || w + 0.01 > 64.0 * P->min_step_x ||
               w + P->row_spread_y + 0.01 > 64.0 * P->min_step_y;
    std::vector<int> xb, yb;
    int warps = P->blk_warps, chunks = P->blk_chunks, rows = P->blk_rows, tw = P->blk_tw, th = P->blk_th;
    // A captured call replays with the shape it was captured with, on the new map's
    // boxes: that shape is kept while it serves the map.
    bool keep = P->captured && rows > 0 && (P->blk_dup || !dup);
    if (keep) {
        xb = boxes(cr, p.n1x, HC * chunks);
        yb = boxes(rr, p.n1y, rows);
        keep = separate(xb, warps) && separate(yb, 1) && widest(xb) - w + WS <= tw && widest(yb) <= th;
    }
    dup = dup || (keep && P->blk_dup);
    const BlkKernel kern = dup ? blk_kernel<true>(w) : blk_kernel<false>(w);
    if (!kern) return ASFD_OK;
    // (process-wide, the same value for every plan)
    ASFD_CUDA(cudaFuncSetAttribute((const void*)kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                   kBlkMaxSmem));
    if (!keep) {
        int dev = 0, sms = 0;
        ASFD_CUDA(cudaGetDevice(&dev));
        ASFD_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
        // columns: 4 warps of one chunk, more warps and then more chunks until
        // blocks two apart are disjoint
        warps = 4;
        chunks = 1;
        for (;;) {
            xb = boxes(cr, p.n1x, HC * chunks);
            if (separate(xb, warps)) break;
            if (warps < kBlkMaxWarps) warps *= 2;
            else if ((long long)HC * chunks * warps < p.n1x) ++chunks;
            else return ASFD_OK;
        }
        tw = widest(xb) - w + WS;
        const auto bytes = [&](int tw_, int th_) {
            return warps * (blk_ring(w) + sizeof(float2) * (size_t)S * tw_ * th_);
        };
        const auto resident = [&](size_t smem, int* per_sm) -> asfd_status {
            ASFD_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(per_sm, (const void*)kern,
                                                                    32 * warps, smem));
            return ASFD_OK;
        };
        const int nc = (int)xb.size() / 2, nbx = (nc + warps - 1) / warps;
        // rows: the fewest for disjoint blocks, then the count that ends soonest
        // by a model in rows: whole waves of resident blocks per colour (a warp
        // waits on its own chain of latencies, so a full SM takes no longer than
        // one block), each of its rows and a fixed part (the empty and the last
        // window, the merge)
        double best = 1e300;
        int best_per_sm = 0;
        asfd_status s;
        rows = 0;
        for (int r = 8; r < 2 * p.n1y; r += std::max(1, r / 8)) {
            const std::vector<int> b = boxes(rr, p.n1y, r);
            if (!separate(b, 1)) continue;
            const int h = widest(b);
            const size_t smem = bytes(tw, h);
            if (smem > kBlkMaxSmem) break;
            int per_sm = 0;
            if ((s = resident(smem, &per_sm)) != ASFD_OK) return s;
            if (per_sm < 1) break;
            const int nby = (int)b.size() / 2;
            double t = 0.0;
            for (int c = 0; c < 4; ++c) {
                const long long blocks = (long long)((nbx + 1 - (c & 1)) / 2) * ((nby + 1 - c / 2) / 2);
                const long long slots = (long long)sms * per_sm;
                t += (double)((blocks + slots - 1) / slots) * (r * chunks + 2.0 * w + 8.0) + 4.0;
            }
            if (t < best) {
                best = t;
                best_per_sm = per_sm;
                rows = r;
                th = h;
                yb = b;
            }
        }
        if (rows == 0) {
            P->blk_rows = 0;
            return ASFD_OK;
        }
        // room for footprints that move by a cell or two in later maps (above),
        // where it costs no resident block
        for (int e = 2; e > 0; --e) {
            int per_sm = 0;
            if (bytes(tw + e, th + e) > kBlkMaxSmem) continue;
            if ((s = resident(bytes(tw + e, th + e), &per_sm)) != ASFD_OK) return s;
            if (per_sm < best_per_sm) continue;
            tw += e;
            th += e;
            break;
        }
    }
    const int ncols = (int)xb.size() / 2;
    asfd_status s;
    if (!P->blk_xbox) {  // sized for the most groups of any height map
        const size_t n = (size_t)((p.n1x + HC - 1) / HC) + (size_t)((p.n1y + 7) / 8);
        if ((s = plan_alloc_buffer(P, reinterpret_cast<void**>(&P->blk_xbox), sizeof(int) * 2 * n)) != ASFD_OK)
            return s;
    }
    xb.insert(xb.end(), yb.begin(), yb.end());
    ASFD_CUDA(cudaMemcpyAsync(P->blk_xbox, xb.data(), sizeof(int) * xb.size(), cudaMemcpyHostToDevice, st));
    ASFD_CUDA(cudaStreamSynchronize(st));
    P->blk_ybox = P->blk_xbox + 2 * ncols;
    P->blk_warps = warps;
    P->blk_chunks = chunks;
    P->blk_rows = rows;
    P->blk_ncols = ncols;
    P->blk_nbx = (ncols + warps - 1) / warps;
    P->blk_nby = (int)yb.size() / 2;
    P->blk_tw = tw;
    P->blk_th = th;
    P->blk_dup = dup;
    P->blk = true;
    return ASFD_OK;
}

asfd_status wide_fold_warp_slots(int w, long long* slots)
{
    int dev = 0, sms = 0, per_sm = 0;
    ASFD_CUDA(cudaGetDevice(&dev));
    ASFD_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    const void* k = nullptr;
    switch (w) {
#define ASFD_FK(W) case W: k = (const void*)spread_fold_kernel<W>; break;
        ASFD_FK(8) ASFD_FK(9) ASFD_FK(10) ASFD_FK(11) ASFD_FK(12) ASFD_FK(13) ASFD_FK(14) ASFD_FK(15)
        ASFD_FK(16)
#undef ASFD_FK
        default: return fail(ASFD_ERR_UNSUPPORTED, "kernel width outside 2..16");
    }
    ASFD_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, 32 * kDenseWarps, 0));
    *slots = (long long)sms * std::max(per_sm, 1) * kDenseWarps;
    return ASFD_OK;
}

cudaError_t launch_wide_fold(const SpreadArgs& a, int w, cudaStream_t st)
{
    const unsigned blocks = (unsigned)((a.dense_items + kDenseWarps - 1) / kDenseWarps);
    switch (w) {
#define ASFD_FL(W) case W: return launch_chained(spread_fold_kernel<W>, blocks, 32 * kDenseWarps, 0, st, a);
        ASFD_FL(8) ASFD_FL(9) ASFD_FL(10) ASFD_FL(11) ASFD_FL(12) ASFD_FL(13) ASFD_FL(14) ASFD_FL(15)
        ASFD_FL(16)
#undef ASFD_FL
        default: return cudaErrorInvalidValue;
    }
}

asfd_status launch_spread_block(asfd_plan_s* P, const float2* u1, cudaStream_t st)
{
    BlkArgs a;
    a.s = make_spread_args(P, u1);
    a.xbox = P->blk_xbox;
    a.ybox = P->blk_ybox;
    a.chunks = P->blk_chunks;
    a.rows = P->blk_rows;
    a.ncols = P->blk_ncols;
    a.nbx = P->blk_nbx;
    a.nby = P->blk_nby;
    a.tw = P->blk_tw;
    a.th = P->blk_th;
    const size_t smem = P->blk_warps * (blk_ring(P->w) +
                                        sizeof(float2) * (size_t)blk_split(P->w) * a.tw * a.th);
    const BlkKernel kern = P->blk_dup ? blk_kernel<true>(P->w) : blk_kernel<false>(P->w);
    for (int c = 0; c < 4; ++c) {
        a.cx = c & 1;
        a.cy = c / 2;
        const dim3 grid((a.nbx + 1 - a.cx) / 2, (a.nby + 1 - a.cy) / 2);
        if (grid.x == 0 || grid.y == 0) continue;
        const cudaError_t e = launch_chained(kern, grid, 32 * P->blk_warps, smem, st, a);
        if (e != cudaSuccess) return cuda_fail(e, "spread_block_kernel launch");
    }
    return ASFD_OK;
}

}  // namespace asfd
