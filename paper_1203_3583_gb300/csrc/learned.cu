// Learned spreading kernel: a per-source-tile tabulated kernel predicted by a
// small MLP from tile features, with a learned correction of the
// deconvolution, trained on the GPU against a reference field.
//
// Kernel.  Width kLearnW (= 4, against 7 for the ES kernel at the same
// target accuracy).  Tap a of axis x of a sample in source tile t has weight
//   P_{t,x,a}(2 dx - 1) = sum_k table[t][x][a][k] (2 dx - 1)^k,  k <= 7,
// where dx in [0, 1) is the sample's offset from its first tap, likewise y.
// table[t] = base + s * MLP(features[t]); base is a shared trainable table
// (initialised by a least-squares fit of the ES kernel of width 4), the MLP
// has one tanh hidden layer, and s = kLearnOutScale.  The deconvolution is
// the ES width-4 one times 1 + sum_j d_j T_{2j}(2 m'/M) per axis (even
// Chebyshev polynomials of the centred destination index), d trainable.
//
// Features of a source tile (dimensionless, so that a model transfers across
// grid sizes): 1, its mean fine-grid position in x and y relative to the grid
// centre (units of nf/2), its mean sample spacing on the fine grid minus one
// in x and y, and 100 x its mean q = d1/(z0 - d1).
//
// Training step (asfd_learned_train_step): loss L = |u2 - ref|^2 / |ref|^2.
//   forward with the current tables -> u2;  g = dL/du2 = 2 (u2 - ref)/|ref|^2
//   dL/dcorr_x[mx] = Re sum_my conj(g) u2 / corr_x[mx]  (likewise y) -> dL/dd
//   b~ = F^H D^H g (the adjoint FFT passes);  for every tap of every sample
//   v = Re[conj(b~_cell) c_n] and dL/dtable[t][x][a][k] += v P_{t,y,b} t_x^k
//   (likewise y); MLP backward over tiles; Adam update; tables refreshed.
// All of it runs in the kernels of this file and the FFT passes; the host only
// sequences launches and reads back the loss.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "asfd_impl.cuh"
#include "fft.cuh"
#include "sample.cuh"
#include "spread.cuh"

namespace asfd {

namespace {

// ---- features (plan time) ---------------------------------------------------

__global__ void __launch_bounds__(256) features_kernel(const float* q, const AxisEntry* ax,
                                                       const AxisEntry* ay, const double* bux,
                                                       const double* buy, int n1x, int n1y,
                                                       int nstx, int nfx, int nfy, float* feat)
{
    const int t = blockIdx.x;
    const int nx = (t % nstx) * kSrcTile + threadIdx.x % kSrcTile;
    const int ny = (t / nstx) * kSrcTile + threadIdx.x / kSrcTile;
    float v[5] = {0.f, 0.f, 0.f, 0.f, 0.f};  // gx, gy, spacing x, spacing y, q
    float cnt[3] = {0.f, 0.f, 0.f};
    if (nx < n1x && ny < n1y) {
        const size_t n = (size_t)ny * n1x + nx;
        const float qq = q[n];
        const double gx = bux[nx] + (double)(ax[nx].s * qq);
        const double gy = buy[ny] + (double)(ay[ny].s * qq);
        v[0] = (float)((gx - 0.5 * nfx) / (0.5 * nfx));
        v[1] = (float)((gy - 0.5 * nfy) / (0.5 * nfy));
        v[4] = qq;
        cnt[0] = 1.f;
        if (nx + 1 < n1x) {
            v[2] = (float)(bux[nx + 1] + (double)(ax[nx + 1].s * q[n + 1]) - gx);
            cnt[1] = 1.f;
        }
        if (ny + 1 < n1y) {
            v[3] = (float)(buy[ny + 1] + (double)(ay[ny + 1].s * q[n + n1x]) - gy);
            cnt[2] = 1.f;
        }
    }
    __shared__ float red[8][8];
    float acc[8] = {v[0], v[1], v[2], v[3], v[4], cnt[0], cnt[1], cnt[2]};
#pragma unroll
    for (int i = 0; i < 8; ++i)
        for (int o = 16; o > 0; o >>= 1) acc[i] += __shfl_xor_sync(0xffffffffu, acc[i], o);
    if ((threadIdx.x & 31) == 0)
        for (int i = 0; i < 8; ++i) red[threadIdx.x / 32][i] = acc[i];
    __syncthreads();
    if (threadIdx.x == 0) {
        float s[8] = {0, 0, 0, 0, 0, 0, 0, 0};
        for (int w = 0; w < 8; ++w)
            for (int i = 0; i < 8; ++i) s[i] += red[w][i];
        const float c0 = fmaxf(s[5], 1.f), c1 = fmaxf(s[6], 1.f), c2 = fmaxf(s[7], 1.f);
        float* f = feat + (size_t)t * kLearnFeat;
        f[0] = 1.f;
        f[1] = s[0] / c0;
        f[2] = s[1] / c0;
        f[3] = (s[6] > 0.f ? s[2] / c1 : 1.f) - 1.f;
        f[4] = (s[7] > 0.f ? s[3] / c2 : 1.f) - 1.f;
        f[5] = 100.f * s[4] / c0;
    }
}

// ---- MLP forward: features -> hidden -> table --------------------------------

// A block takes kMlpTiles tiles: thread (g, o) holds row o of W2 in registers
// and forms table entry o of the tiles g, g + 4, ...  (One block of 64
// threads per tile read the 8 KB of W2 again for every tile, a cache line per
// lane: 121 us for 16384 tiles; see learned_gradient.)
constexpr int kMlpTiles = 32;

__global__ void __launch_bounds__(256) mlp_forward_kernel(const float* prm, const float* feat,
                                                          int ntiles, float* hid, float* tab)
{
    constexpr int O = kLearnTableSize, H = kLearnHidden, F = kLearnFeat, T = kMlpTiles;
    static_assert(O == 64 && H % 4 == 0, "four tiles at a time in 256 threads");
    __shared__ float w1[H][F + 1], f[T][F];
    __shared__ __align__(16) float h[T][H];
    chain_next();
    chain_wait();
    const int tid = threadIdx.x, t0 = blockIdx.x * T, nt = min(T, ntiles - t0);
    for (int i = tid; i < H * F; i += 256) w1[i / F][i % F] = prm[kLpW1 + i];
    for (int i = tid; i < nt * F; i += 256) f[i / F][i % F] = feat[(size_t)t0 * F + i];
    const int o = tid % O;
    float w2[H];
#pragma unroll
    for (int i = 0; i < H; ++i) w2[i] = prm[kLpW2 + o * H + i];
    const float b2 = prm[kLpB2 + o], base = prm[kLpBase + o];
    __syncthreads();
    for (int i = tid; i < nt * H; i += 256) {
        const int t = i / H, k = i % H;
        float s = prm[kLpB1 + k];
#pragma unroll
        for (int j = 0; j < F; ++j) s = fmaf(w1[k][j], f[t][j], s);
        const float hv = tanhf(s);
        h[t][k] = hv;
        hid[(size_t)t0 * H + i] = hv;
    }
    __syncthreads();
    for (int t = tid / O; t < nt; t += 256 / O) {
        float s = b2;
        const float4* h4 = reinterpret_cast<const float4*>(h[t]);
#pragma unroll
        for (int i = 0; i < H / 4; ++i) {
            const float4 v = h4[i];
            s = fmaf(w2[4 * i], v.x, s);
            s = fmaf(w2[4 * i + 1], v.y, s);
            s = fmaf(w2[4 * i + 2], v.z, s);
            s = fmaf(w2[4 * i + 3], v.w, s);
        }
        tab[(size_t)(t0 + t) * O + o] = base + kLearnOutScale * s;
    }
}

// ---- deconvolution correction ----------------------------------------------

// T_{2j}(u) for j = 1..kLearnCheb
__device__ __forceinline__ void cheb_even(float u, float (&T)[kLearnCheb])
{
    float t0 = 1.f, t1 = u;
    for (int n = 2, j = 0; j < kLearnCheb; ++n) {
        const float t2 = 2.f * u * t1 - t0;
        t0 = t1;
        t1 = t2;
        if ((n & 1) == 0) T[j++] = t2;
    }
}

__global__ void deconv_build_kernel(const float* prm, const float2* cb, float2* c, float* corr, int m,
                                    int off)
{
    chain_next();
    chain_wait();
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= m) return;
    const float u = 2.f * (float)(k - m / 2) / (float)m;
    float T[kLearnCheb];
    cheb_even(u, T);
    float s = 1.f;
    for (int j = 0; j < kLearnCheb; ++j) s = fmaf(prm[off + j], T[j], s);
    corr[k] = s;
    c[k] = make_float2(cb[k].x * s, cb[k].y * s);
}

// ---- loss --------------------------------------------------------------------

constexpr int kLossBlocks = 1216;  // eight per SM

// sum + err += v on a pair, err collecting the rounding errors of sum exactly
// (Knuth's two-sum)
__device__ __forceinline__ void two_sum2(float2& sum, float2& err, float2 v)
{
    const float2 s = cadd(sum, v);
    const float2 b = csub(s, sum);
    err = cadd(err, cadd(csub(sum, csub(s, b)), csub(v, b)));
    sum = s;
}

// sum + err += (v + dv)^2 on a pair, exactly but for the last term's rounding
__device__ __forceinline__ void add_square2(float2& sum, float2& err, float2 v, float2 dv)
{
    const float2 p = mul_f2(v, v);
    const float2 pe = fma_f2(v, v, make_float2(-p.x, -p.y));
    two_sum2(sum, err, p);
    err = cadd(err, fma_f2(cadd(v, v), dv, pe));
}

// Whether a thread's FP32 sum of squares is exact to about 2^-40: not so
// large that a term may have overflowed, nor so small that the terms'
// rounding errors have underflowed (the caller then sums again in FP64).
__device__ __forceinline__ bool squares_in_range(float2 sum)
{
    const float t = sum.x + sum.y;
    return t > 8.2718061e-25f && t < 1.2676506e30f;  // 2^-80 .. 2^100
}

// Adds the block's sum to *out.  `part`: a slot per thread (256); one warp adds
// them (a shuffle tree in every warp is seven times as many FP64 additions, at
// 2 lanes per clock).  Has a block barrier.
__device__ __forceinline__ void block_add(double v, double* part, double* out)
{
    part[threadIdx.x] = v;
    __syncthreads();
    if (threadIdx.x >= 32) return;
    for (int w = 1; w < 8; ++w) v += part[threadIdx.x + 32 * w];
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (threadIdx.x == 0) atomicAdd(out, v);
}

// red[1] += |ref|^2, and the deconvolution gradients are set to zero.  The
// squares are carried as FP32 values with their exact rounding errors: FP64
// sums over 4.2 M points are bound by the FP64 pipe (this and the squared
// error together took 116 us).
__global__ void __launch_bounds__(256) ref_norm_kernel(const float2* ref, size_t n, double* red,
                                                       float* gcorr, int ncorr)
{
    chain_next();
    chain_wait();
    const size_t i0 = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    const size_t step = (size_t)gridDim.x * blockDim.x;
    for (size_t i = i0; i < (size_t)ncorr; i += step) gcorr[i] = 0.f;
    float2 sum = make_float2(0.f, 0.f), err = sum;
#pragma unroll 8
    for (size_t i = i0; i < n; i += step)
        add_square2(sum, err, ref[i], make_float2(0.f, 0.f));
    double v = ((double)sum.x + (double)sum.y) + ((double)err.x + (double)err.y);
    if (!squares_in_range(sum)) {
        v = 0.0;
        for (size_t i = i0; i < n; i += step) {
            const float2 b = ref[i];
            v += (double)b.x * b.x + (double)b.y * b.y;
        }
    }
    __shared__ double part[256];
    block_add(v, part, red + 1);
}

// One pass over the output: g = dL/du2 = 2 (u2 - ref)/|ref|^2, red[0] +=
// |u2 - ref|^2, and dL/dcorr of both axes (sums of Re[conj(g) u2] / corr over
// the columns' rows and the rows' columns).  A warp takes 128 columns (4 a
// lane) of every 8th row of its block's kLossRows rows.  Four kernels (the
// loss in FP64, g with an FP64 division per point, one pass per axis) took
// 212 us at 2048^2; see learned_gradient.
constexpr int kLossCols = 128, kLossRows = 32;

__global__ void __launch_bounds__(256)
loss_kernel(const float2* u2, const float2* ref, const float* corr, int m2x, int m2y, double* red,
            float2* g, float* gcorr)
{
    chain_next();
    chain_wait();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int c0 = blockIdx.x * kLossCols + lane;
    const int y1 = min(m2y, (int)(blockIdx.y + 1) * kLossRows);
    const float sc = (float)(2.0 / fmax(red[1], 1e-300));
    float2 sum = make_float2(0.f, 0.f), err = sum;
    float col[kLossCols / 32];
#pragma unroll
    for (int j = 0; j < kLossCols / 32; ++j) col[j] = 0.f;
    for (int y = blockIdx.y * kLossRows + warp; y < y1; y += 8) {
        const size_t row = (size_t)y * m2x;
        float across = 0.f;
        float2 us[kLossCols / 32], rs[kLossCols / 32];  // all loads before the first store
#pragma unroll
        for (int j = 0; j < kLossCols / 32; ++j) {
            const int c = c0 + 32 * j;
            us[j] = c < m2x ? u2[row + c] : make_float2(0.f, 0.f);
            rs[j] = c < m2x ? ref[row + c] : make_float2(0.f, 0.f);
        }
#pragma unroll
        for (int j = 0; j < kLossCols / 32; ++j) {
            const int c = c0 + 32 * j;
            if (c < m2x) {
                const float2 a = us[j], b = rs[j];
                // a - b = d + e exactly
                const float2 d = csub(a, b), z = csub(d, a);
                const float2 e = csub(csub(a, csub(d, z)), cadd(b, z));
                add_square2(sum, err, d, e);
                const float2 v = make_float2(sc * d.x, sc * d.y);
                g[row + c] = v;
                const float dot = v.x * a.x + v.y * a.y;
                col[j] += dot;
                across += dot;
            }
        }
        for (int o = 16; o > 0; o >>= 1) across += __shfl_xor_sync(0xffffffffu, across, o);
        if (lane == 0) atomicAdd(&gcorr[m2x + y], across / corr[m2x + y]);
    }
    __shared__ float cols[8][kLossCols];
#pragma unroll
    for (int j = 0; j < kLossCols / 32; ++j) cols[warp][lane + 32 * j] = col[j];
    double e2 = ((double)sum.x + (double)sum.y) + ((double)err.x + (double)err.y);
    if (!squares_in_range(sum)) {
        e2 = 0.0;
        for (int y = blockIdx.y * kLossRows + warp; y < y1; y += 8)
            for (int c = c0; c < min(m2x, (int)(blockIdx.x + 1) * kLossCols); c += 32) {
                const float2 a = u2[(size_t)y * m2x + c], b = ref[(size_t)y * m2x + c];
                const double dx = (double)a.x - b.x, dy = (double)a.y - b.y;
                e2 += dx * dx + dy * dy;
            }
    }
    __shared__ double part[256];
    block_add(e2, part, red);
    const int c = blockIdx.x * kLossCols + threadIdx.x;
    if (threadIdx.x < kLossCols && c < m2x) {
        float t = 0.f;
        for (int w = 0; w < 8; ++w) t += cols[w][threadIdx.x];
        atomicAdd(&gcorr[c], t / corr[c]);
    }
}

// dL/dd_j = sum_k dL/dcorr[k] T_2j(u_k): block 0 the x axis, block 1 the y axis
__global__ void __launch_bounds__(1024) cheb_grad_kernel(const float* gcorr, int m2x, int m2y,
                                                         float* grad)
{
    chain_next();
    chain_wait();
    const int m = blockIdx.x == 0 ? m2x : m2y;
    if (blockIdx.x == 1) gcorr += m2x;
    grad += blockIdx.x == 0 ? kLpDx : kLpDy;
    float s[kLearnCheb];
    for (int j = 0; j < kLearnCheb; ++j) s[j] = 0.f;
    for (int k = threadIdx.x; k < m; k += blockDim.x) {
        const float u = 2.f * (float)(k - m / 2) / (float)m;
        float T[kLearnCheb];
        cheb_even(u, T);
        for (int j = 0; j < kLearnCheb; ++j) s[j] = fmaf(gcorr[k], T[j], s[j]);
    }
    __shared__ float red[kLearnCheb][32];
    for (int j = 0; j < kLearnCheb; ++j) {
        float v = s[j];
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if ((threadIdx.x & 31) == 0) red[j][threadIdx.x / 32] = v;
    }
    __syncthreads();
    if (threadIdx.x < kLearnCheb) {
        float t = 0.f;
        for (int w = 0; w < (int)(blockDim.x / 32); ++w) t += red[threadIdx.x][w];
        grad[threadIdx.x] = t;
    }
}

// ---- dL/dtable from the adjoint grid ------------------------------------------

struct TGArgs {
    const float2* u1;
    const float* q;
    const AxisEntry* ax;
    const AxisEntry* ay;
    const AxisPos* px;
    const AxisPos* py;
    const float2* grid;   // b~ = F^H D^H g over the band
    const float* tab;
    float* tgrad;
    int n1x, n1y, nstx, nfx, nfy;
    float half_w;
    float inc_d;
};

// A warp per source tile, a lane per half column (8 samples): the lane sums its
// samples' contributions to the 64 table entries, per axis and tap the sum
// over the other axis' taps first, then times the powers of t; the warp's 64
// sums meet in one reduce-scatter per tile.  (A thread per sample, with the
// powers inside the 16 taps and a reduce-scatter per 32 samples, took 147 us at
// 2048^2; see learned_gradient.)
constexpr int kTgWarps = 4;

template <bool WRAP>
__global__ void __launch_bounds__(32 * kTgWarps) table_grad_kernel(TGArgs a, int ntiles)
{
    constexpr int W = kLearnW, K = kLearnCoef;
    static_assert(kSrcTile == 16 && 2 * W * K == 64, "half a column per lane, 64 sums over 32 lanes");
    __shared__ __align__(16) float tsm[kTgWarps][2 * W * K];
    chain_next();
    chain_wait();
    const int lane = threadIdx.x & 31, wid = threadIdx.x / 32;
    const int t = blockIdx.x * kTgWarps + wid;
    if (t >= ntiles) return;  // warp-uniform
    // the tile's polynomials as (x, y) coefficient pairs
#pragma unroll
    for (int e = lane; e < 2 * W * K; e += 32)
        tsm[wid][2 * (e % (W * K)) + e / (W * K)] = a.tab[(size_t)t * kLearnTableSize + e];
    __syncwarp();
    const int nx = (t % a.nstx) * kSrcTile + (lane & 15);
    const int ny0 = (t / a.nstx) * kSrcTile + (lane >> 4) * (kSrcTile / 2);
    const int rows = nx < a.n1x ? min(kSrcTile / 2, a.n1y - ny0) : 0;
    const int mx = a.nfx - 1, my = a.nfy - 1;
    float2 G[W][K];  // (x, y) sums
#pragma unroll
    for (int i = 0; i < W; ++i)
#pragma unroll
        for (int k = 0; k < K; ++k) G[i][k] = make_float2(0.f, 0.f);
    Raw next;
    if (rows > 0) next = load_raw(a, nx, ny0);
    for (int r = 0; r < rows; ++r) {
        const Raw s = next;
        if (r + 1 < rows) {  // the next sample's inputs, while this one is processed
            const int ny = ny0 + r + 1;
            const size_t n = (size_t)ny * a.n1x + nx;
            next.q = __ldg(&a.q[n]);
            next.u = a.u1[n];
            next.ey = a.ay[ny];
            next.py = a.py[ny];
        }
        int l0x, l0y;
        float dx, dy;
        sample_pos(s.ex, s.ey, s.px, s.py, s.q, a.half_w, l0x, l0y, dx, dy);
        float2 B[W][W];
        if constexpr (WRAP) {
#pragma unroll
            for (int b = 0; b < W; ++b) {
                const float2* row = a.grid + (size_t)((l0y + b) & my) * a.nfx;
#pragma unroll
                for (int i = 0; i < W; ++i) B[b][i] = row[(l0x + i) & mx];
            }
        } else {
            // (clamped all the same: every address stays inside the grid)
            const float2* cell = a.grid + (size_t)min(max(l0y, 0), a.nfy - W) * a.nfx +
                                 min(max(l0x, 0), a.nfx - W);
#pragma unroll
            for (int b = 0; b < W; ++b)
#pragma unroll
                for (int i = 0; i < W; ++i) B[b][i] = cell[(size_t)b * a.nfx + i];
        }
        const float2 c = sample_value_fast(s, a.inc_d);
        float wx[W], wy[W];
        table_weights_smem<W>(reinterpret_cast<const float4*>(tsm[wid]), dx, dy, wx, wy);
        // sums of the cells over the other axis' taps, then Re[conj(sum) c]
        float2 vc[W], vr[W];
#pragma unroll
        for (int b = 0; b < W; ++b) {
            vr[b] = mul2(B[b][0], wx[0]);
#pragma unroll
            for (int i = 1; i < W; ++i) vr[b] = fma2(B[b][i], wx[i], vr[b]);
#pragma unroll
            for (int i = 0; i < W; ++i) vc[i] = b == 0 ? mul2(B[b][i], wy[b]) : fma2(B[b][i], wy[b], vc[i]);
        }
        const float2 tt = make_float2(fmaf(2.f, dx, -1.f), fmaf(2.f, dy, -1.f));
        float2 pw[K];
        pw[0] = make_float2(1.f, 1.f);
#pragma unroll
        for (int k = 1; k < K; ++k) pw[k] = mul_f2(pw[k - 1], tt);
#pragma unroll
        for (int i = 0; i < W; ++i) {
            const float2 v = make_float2(vc[i].x * c.x + vc[i].y * c.y, vr[i].x * c.x + vr[i].y * c.y);
#pragma unroll
            for (int k = 0; k < K; ++k) G[i][k] = fma_f2(v, pw[k], G[i][k]);
        }
    }
    // reduce-scatter by recursive halving: at offset o a lane keeps the half
    // of its values selected by lane bit o and adds its partner's copy of
    // that half; lane l ends with the warp's sums of entries 2l and 2l + 1
    float v[64];
#pragma unroll
    for (int i = 0; i < W; ++i)
#pragma unroll
        for (int k = 0; k < K; ++k) {
            v[i * K + k] = G[i][k].x;
            v[(W + i) * K + k] = G[i][k].y;
        }
#pragma unroll
    for (int lvl = 0; lvl < 5; ++lvl) {
        const int o = 16 >> lvl, half = 32 >> lvl;
        const bool upper = (lane & o) != 0;
#pragma unroll
        for (int i = 0; i < half; ++i) {
            const float send = upper ? v[i] : v[i + half];
            const float keep = upper ? v[i + half] : v[i];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
        }
    }
    reinterpret_cast<float2*>(a.tgrad + (size_t)t * kLearnTableSize)[lane] = make_float2(v[0], v[1]);
}

// ---- MLP backward over tiles (block-private accumulation, then atomics) --------

// Blocks walk over groups of kBackTiles tiles.  A thread keeps its 8 entries of
// dL/dW2 (row o, 8 columns), its entry of dL/dW1 and of the biases in
// registers over all groups, and column ti of W2 for the hidden gradient of
// its (tile, unit) in each group; the next group's inputs are loaded while one
// is processed.  (One tile at a time, with the sums in shared memory and 32 of
// 256 threads on the hidden gradient, took 92 us for 16384 tiles; see
// learned_gradient.)
constexpr int kBackTiles = 8;
constexpr int kBackBlocks = 304;      // two per SM
constexpr int kMlpParams = kLpDx;     // table and MLP parameters come first

__global__ void __launch_bounds__(256) mlp_backward_kernel(const float* prm, const float* feat,
                                                           const float* hid, const float* tgrad,
                                                           int ntiles, float* part)
{
    constexpr int O = kLearnTableSize, H = kLearnHidden, F = kLearnFeat, T = kBackTiles;
    static_assert(T * H == 256 && T * O == 512 && O * H == 8 * 256 && H * F <= 256,
                  "one (tile, unit) per thread");
    __shared__ __align__(16) float dout[T][O], h[T][H];
    __shared__ float f[T][F], dh[T][H];
    chain_next();
    chain_wait();
    const int tid = threadIdx.x;
    const int o = tid / 4, i0 = (tid % 4) * 8;  // this thread's entries of W2
    const int k1 = tid / F, j1 = tid % F;       // and of W1 (tid < H F)
    const int tt = tid / H, ti = tid % H;       // its hidden gradient
    float w2[O];
#pragma unroll
    for (int k = 0; k < O; ++k) w2[k] = prm[kLpW2 + k * H + ti];
    float gw2[8], gw1 = 0.f, gb1 = 0.f, gbase = 0.f;
#pragma unroll
    for (int i = 0; i < 8; ++i) gw2[i] = 0.f;
    // this thread's inputs of a group: two table gradients (entry tid % O of
    // tiles tid / O and tid / O + 4), one hidden value, one feature
    float n0, n1, nh, nf;
    auto fetch = [&](int t0) {
        const int nt = min(T, ntiles - t0);
        n0 = tid < nt * O ? tgrad[(size_t)t0 * O + tid] : 0.f;
        n1 = tid + 256 < nt * O ? tgrad[(size_t)t0 * O + tid + 256] : 0.f;
        nh = tid < nt * H ? hid[(size_t)t0 * H + tid] : 0.f;
        nf = tid < nt * F ? feat[(size_t)t0 * F + tid] : 0.f;
    };
    fetch(blockIdx.x * T);
    for (int t0 = blockIdx.x * T; t0 < ntiles; t0 += gridDim.x * T) {
        __syncthreads();  // the previous group's readers are done
        gbase += n0 + n1;
        dout[tid / O][tid % O] = kLearnOutScale * n0;
        dout[tid / O + 4][tid % O] = kLearnOutScale * n1;
        h[tt][ti] = nh;
        if (tid < T * F) f[tid / F][tid % F] = nf;
        const float hv = nh;
        __syncthreads();
        if (t0 + gridDim.x * T < ntiles) fetch(t0 + gridDim.x * T);
        float s0 = 0.f, s1 = 0.f, s2 = 0.f, s3 = 0.f;
        const float4* d4 = reinterpret_cast<const float4*>(dout[tt]);
#pragma unroll
        for (int k = 0; k < O / 4; ++k) {
            const float4 d = d4[k];
            s0 = fmaf(w2[4 * k], d.x, s0);
            s1 = fmaf(w2[4 * k + 1], d.y, s1);
            s2 = fmaf(w2[4 * k + 2], d.z, s2);
            s3 = fmaf(w2[4 * k + 3], d.w, s3);
        }
        dh[tt][ti] = ((s0 + s1) + (s2 + s3)) * (1.f - hv * hv);
#pragma unroll
        for (int t = 0; t < T; ++t) {
            const float d = dout[t][o];
            const float4 a = *reinterpret_cast<const float4*>(&h[t][i0]);
            const float4 b = *reinterpret_cast<const float4*>(&h[t][i0 + 4]);
            gw2[0] = fmaf(d, a.x, gw2[0]);
            gw2[1] = fmaf(d, a.y, gw2[1]);
            gw2[2] = fmaf(d, a.z, gw2[2]);
            gw2[3] = fmaf(d, a.w, gw2[3]);
            gw2[4] = fmaf(d, b.x, gw2[4]);
            gw2[5] = fmaf(d, b.y, gw2[5]);
            gw2[6] = fmaf(d, b.z, gw2[6]);
            gw2[7] = fmaf(d, b.w, gw2[7]);
        }
        __syncthreads();
        if (tid < H * F) {
#pragma unroll
            for (int t = 0; t < T; ++t) gw1 = fmaf(dh[t][k1], f[t][j1], gw1);
        }
        if (tid < H) {
#pragma unroll
            for (int t = 0; t < T; ++t) gb1 += dh[t][tid];
        }
    }
    float* out = part + (size_t)blockIdx.x * kMlpParams;
#pragma unroll
    for (int i = 0; i < 8; ++i) out[kLpW2 + o * H + i0 + i] = gw2[i];
    if (tid < H * F) out[kLpW1 + tid] = gw1;
    if (tid < H) out[kLpB1 + tid] = gb1;
    __syncthreads();
    float* base = &dout[0][0];  // [4][O]
    base[tid] = gbase;
    __syncthreads();
    if (tid < O) {
        const float v = (base[tid] + base[tid + O]) + (base[tid + 2 * O] + base[tid + 3 * O]);
        out[kLpBase + tid] = v;
        out[kLpB2 + tid] = kLearnOutScale * v;
    }
}

// The blocks' sums, added in order: a thread per parameter and eighth of the
// blocks.
__global__ void __launch_bounds__(256) mlp_reduce_kernel(const float* part, int blocks, float* grad)
{
    __shared__ float red[8][32];
    chain_next();
    chain_wait();
    const int lane = threadIdx.x & 31, wid = threadIdx.x / 32;
    const int i = blockIdx.x * 32 + lane;
    float v = 0.f;
    if (i < kMlpParams) {
#pragma unroll 8
        for (int b = wid; b < blocks; b += 8) v += part[(size_t)b * kMlpParams + i];
    }
    red[wid][lane] = v;
    __syncthreads();
    if (wid == 0 && i < kMlpParams) {
        for (int w = 1; w < 8; ++w) v += red[w][lane];
        grad[i] = v;
    }
}


__global__ void adam_kernel(float* p, const float* g, float* m, float* v, int n, float lr, float b1, float b2, float c1,
                            float c2, float eps)
{
    chain_next();
    chain_wait();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    p[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
}

// ---- host helpers ------------------------------------------------------------

// Least-squares fit (FP64 normal equations on Chebyshev nodes) of the ES
// kernel of width kLearnW, tap by tap, by polynomials of degree kLearnDeg in
// t = 2 dx - 1: the initial shared table.
void fit_es_table(double beta, std::vector<float>& table)
{
    constexpr int W = kLearnW, K = kLearnCoef, NP = 256;
    const double pi = 3.14159265358979323846;
    table.assign(kLearnTableSize, 0.f);
    for (int a = 0; a < W; ++a) {
        double A[K][K] = {}, b[K] = {};
        for (int p = 0; p < NP; ++p) {
            const double t = std::cos(pi * (p + 0.5) / NP);
            const double dx = 0.5 * (t + 1.0);
            const double z = dx + a - 0.5 * W;
            const double u = 2.0 * z / W;
            const double psi = std::exp(beta * (std::sqrt(std::max(0.0, 1.0 - u * u)) - 1.0));
            double pw[K];
            pw[0] = 1.0;
            for (int k = 1; k < K; ++k) pw[k] = pw[k - 1] * t;
            for (int i = 0; i < K; ++i) {
                b[i] += pw[i] * psi;
                for (int j = 0; j < K; ++j) A[i][j] += pw[i] * pw[j];
            }
        }
        // Gaussian elimination with partial pivoting
        for (int c = 0; c < K; ++c) {
            int piv = c;
            for (int r = c + 1; r < K; ++r)
                if (std::fabs(A[r][c]) > std::fabs(A[piv][c])) piv = r;
            for (int j = 0; j < K; ++j) std::swap(A[c][j], A[piv][j]);
            std::swap(b[c], b[piv]);
            for (int r = c + 1; r < K; ++r) {
                const double f = A[r][c] / A[c][c];
                for (int j = c; j < K; ++j) A[r][j] -= f * A[c][j];
                b[r] -= f * b[c];
            }
        }
        double x[K];
        for (int c = K - 1; c >= 0; --c) {
            double s = b[c];
            for (int j = c + 1; j < K; ++j) s -= A[c][j] * x[j];
            x[c] = s / A[c][c];
        }
        for (int k = 0; k < K; ++k) {
            table[(0 * W + a) * K + k] = (float)x[k];
            table[(1 * W + a) * K + k] = (float)x[k];
        }
    }
}

}  // namespace

asfd_status learned_features(asfd_plan_s* P, cudaStream_t st)
{
    const int nst = P->nstx * P->nsty;
    features_kernel<<<nst, kSrcTile * kSrcTile, 0, st>>>(P->q, P->ax, P->ay, P->bux, P->buy,
                                                        P->prm.n1x, P->prm.n1y, P->nstx, P->nfx,
                                                        P->nfy, P->lfeat);
    ASFD_CUDA(cudaGetLastError());
    return ASFD_OK;
}

asfd_status learned_refresh(asfd_plan_s* P, cudaStream_t st)
{
    const int nst = P->nstx * P->nsty;
    using F = const float*;
    ASFD_CUDA(launch_chained(mlp_forward_kernel, dim3((nst + kMlpTiles - 1) / kMlpTiles), 256, 0, st,
                             F(P->lparams), F(P->lfeat), nst, P->lhid, P->ltab));
    const int m2x = P->prm.m2x, m2y = P->prm.m2y;
    ASFD_CUDA(launch_chained(deconv_build_kernel, dim3((m2x + 255) / 256), 256, 0, st, F(P->lparams),
                             (const float2*)P->cxb, P->cx, P->lcorr, m2x, kLpDx));
    ASFD_CUDA(launch_chained(deconv_build_kernel, dim3((m2y + 255) / 256), 256, 0, st, F(P->lparams),
                             (const float2*)P->cyb, P->cy, P->lcorr + m2x, m2y, kLpDy));
    // no kernel queued after this starts before the tables are complete (it would
    // before a chained launch): the column pass reads cx and cy as constants
    ASFD_CUDA(cudaMemsetAsync(P->lred + 2, 0, sizeof(double), st));
    return ASFD_OK;
}

asfd_status learned_init(asfd_plan_s* P, cudaStream_t st)
{
    const int nst = P->nstx * P->nsty;
    const int mm = P->prm.m2x + P->prm.m2y;
    auto A = [&](void** p, size_t bytes) { return plan_alloc_buffer(P, p, bytes); };
    asfd_status s;
#define LA(ptr, bytes) if ((s = A(reinterpret_cast<void**>(&P->ptr), (bytes))) != ASFD_OK) return s
    LA(ltab, sizeof(float) * nst * kLearnTableSize);
    LA(lfeat, sizeof(float) * nst * kLearnFeat);
    LA(lhid, sizeof(float) * nst * kLearnHidden);
    LA(ltgrad, sizeof(float) * nst * kLearnTableSize);
    LA(lparams, sizeof(float) * kLearnParams);
    LA(lgrad, sizeof(float) * kLearnParams);
    LA(lm, sizeof(float) * kLearnParams);
    LA(lv, sizeof(float) * kLearnParams);
    LA(cxb, sizeof(float2) * P->prm.m2x);
    LA(cyb, sizeof(float2) * P->prm.m2y);
    LA(lcorr, sizeof(float) * mm);
    LA(lcgrad, sizeof(float) * mm);
    LA(lred, sizeof(double) * 3);
    LA(lpart, sizeof(float) * kBackBlocks * kMlpParams);
#undef LA
    // the ES width-4 deconvolution/chirp tables become the base tables
    ASFD_CUDA(cudaMemcpyAsync(P->cxb, P->cx, sizeof(float2) * P->prm.m2x, cudaMemcpyDeviceToDevice, st));
    ASFD_CUDA(cudaMemcpyAsync(P->cyb, P->cy, sizeof(float2) * P->prm.m2y, cudaMemcpyDeviceToDevice, st));
    // initial parameters: fitted base table, small seeded W1, zero elsewhere
    std::vector<float> h(kLearnParams, 0.f), base;
    fit_es_table(P->beta, base);
    for (int i = 0; i < kLearnTableSize; ++i) h[kLpBase + i] = base[i];
    unsigned long long st64 = 0x9E3779B97F4A7C15ull;
    for (int i = 0; i < kLearnHidden * kLearnFeat; ++i) {
        st64 = st64 * 6364136223846793005ull + 1442695040888963407ull;
        const float u = (float)((st64 >> 40) & 0xFFFFFF) / 16777216.0f;
        h[kLpW1 + i] = 0.5f * (2.f * u - 1.f);
    }
    ASFD_CUDA(cudaMemcpyAsync(P->lparams, h.data(), sizeof(float) * kLearnParams,
                              cudaMemcpyHostToDevice, st));
    ASFD_CUDA(cudaMemsetAsync(P->lm, 0, sizeof(float) * kLearnParams, st));
    ASFD_CUDA(cudaMemsetAsync(P->lv, 0, sizeof(float) * kLearnParams, st));
    P->lstep = 0;
    s = learned_features(P, st);
    if (s != ASFD_OK) return s;
    s = learned_refresh(P, st);
    if (s != ASFD_OK) return s;
    ASFD_CUDA(cudaStreamSynchronize(st));  // h must outlive the copy
    return ASFD_OK;
}

// Forward with the current model, loss against `ref`, and every parameter
// gradient into P->lgrad (no update).  Kernel times at 2048^2 samples and
// points (CUDA events of a trace; before -> now, us): loss, residual and
// deconvolution gradients 212 -> 41 (ref_norm 13.8, loss 27.4: bound by memory,
// 134 MB), both Chebyshev sums 14.3 -> 4.2, table gradients 147 -> 68 (half the
// issue slots; 128 registers leave 16 warps per SM), MLP backward 92 -> 18
// (with its reduction), MLP forward 121 -> not run here; the whole call 851 ->
// 374 us.
asfd_status learned_gradient(asfd_plan_s* P, const float2* u1, const float2* ref, cudaStream_t st)
{
    const int nst = P->nstx * P->nsty;
    const int m2x = P->prm.m2x, m2y = P->prm.m2y;
    const size_t m = (size_t)m2x * m2y;
    asfd_status s;
    // forward with the current model (its tables are current: every change of
    // the parameters or the height map rebuilds them)
    // (the memset first: it would break the chain of the kernels' launches)
    ASFD_CUDA(cudaMemsetAsync(P->lred, 0, sizeof(double) * 2, st));
    if ((s = launch_spread(P, u1, st)) != ASFD_OK) return s;
    if ((s = launch_fft_rows(P, st)) != ASFD_OK) return s;
    if ((s = launch_fft_cols(P, P->lu2, st)) != ASFD_OK) return s;
    // loss, its gradient with respect to u2 and the deconvolution correction's
    using F = const float*;
    using F2 = const float2*;
    ASFD_CUDA(launch_chained(ref_norm_kernel, dim3(kLossBlocks), 256, 0, st, ref, m, P->lred, P->lcgrad,
                             m2x + m2y));
    ASFD_CUDA(launch_chained(loss_kernel,
                             dim3((m2x + kLossCols - 1) / kLossCols, (m2y + kLossRows - 1) / kLossRows),
                             256, 0, st, F2(P->lu2), ref, F(P->lcorr), m2x, m2y, P->lred, P->lres,
                             P->lcgrad));
    ASFD_CUDA(launch_chained(cheb_grad_kernel, dim3(2), 1024, 0, st, F(P->lcgrad), m2x, m2y, P->lgrad));
    // table gradients through the adjoint grid
    if ((s = launch_fft_cols_adj(P, P->lres, st)) != ASFD_OK) return s;
    if ((s = launch_fft_rows_adj(P, st)) != ASFD_OK) return s;
    TGArgs a;
    a.u1 = u1;
    a.q = P->q;
    a.ax = P->ax;
    a.ay = P->ay;
    a.px = P->px;
    a.py = P->py;
    a.grid = P->grid;
    a.tab = P->ltab;
    a.tgrad = P->ltgrad;
    a.n1x = P->prm.n1x;
    a.n1y = P->prm.n1y;
    a.nstx = P->nstx;
    a.nfx = P->nfx;
    a.nfy = P->nfy;
    a.half_w = 0.5f * kLearnW;
    a.inc_d = (float)P->inc_d;
    const unsigned tgb = (unsigned)((nst + kTgWarps - 1) / kTgWarps);
    ASFD_CUDA(launch_chained(P->wraps ? table_grad_kernel<true> : table_grad_kernel<false>, dim3(tgb),
                             32 * kTgWarps, 0, st, a, nst));
    const int groups = std::min((nst + kBackTiles - 1) / kBackTiles, kBackBlocks);
    ASFD_CUDA(launch_chained(mlp_backward_kernel, dim3(groups), 256, 0, st, F(P->lparams), F(P->lfeat),
                             F(P->lhid), F(P->ltgrad), nst, P->lpart));
    ASFD_CUDA(launch_chained(mlp_reduce_kernel, dim3((kMlpParams + 31) / 32), 256, 0, st, F(P->lpart),
                             groups, P->lgrad));
    return ASFD_OK;
}

asfd_status learned_read_loss(asfd_plan_s* P, double* loss_out, cudaStream_t st)
{
    double red[2];
    ASFD_CUDA(cudaMemcpyAsync(red, P->lred, sizeof(red), cudaMemcpyDeviceToHost, st));
    ASFD_CUDA(cudaStreamSynchronize(st));
    *loss_out = red[0] / (red[1] > 0.0 ? red[1] : 1.0);
    return ASFD_OK;
}

asfd_status learned_train_step(asfd_plan_s* P, const float2* u1, const float2* ref, float lr,
                               double* loss_out, cudaStream_t st)
{
    asfd_status s = learned_gradient(P, u1, ref, st);
    if (s != ASFD_OK) return s;
    // Adam
    ++P->lstep;
    const float b1 = 0.9f, b2 = 0.999f;
    const float c1 = 1.f - std::pow(b1, (float)P->lstep), c2 = 1.f - std::pow(b2, (float)P->lstep);
    ASFD_CUDA(launch_chained(adam_kernel, dim3((kLearnParams + 255) / 256), 256, 0, st, P->lparams,
                             (const float*)P->lgrad, P->lm, P->lv, kLearnParams, lr, b1, b2, c1, c2, 1e-12f));
    if ((s = learned_refresh(P, st)) != ASFD_OK) return s;
    if (loss_out) return learned_read_loss(P, loss_out, st);
    return ASFD_OK;
}

}  // namespace asfd
