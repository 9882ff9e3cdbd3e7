// Adjoint (type-2) of the forward transform, for gradients of a real loss.
//
// The forward map is u2 = D F S c with c_n = u1_n E_n (E_n = exp(i theta_n),
// the prefactor of Eq. 8), S the spread with the ES kernel at the fine-grid
// position G_n of each sample, F the 2D DFT restricted to the kept bins and D
// the diagonal deconvolution / destination chirp / global factor (Eq. 8).
// Given gu2 = dL/dRe(u2) + i dL/dIm(u2):
//   b~ = F^H D^H gu2          (two inverse-sign FFT passes, fft.cu)
//   I0 = sum_s psi(s - G) b~_s,  I_a = sum_s psi'(s_a - G_a) psi(s_b - G_b) b~_s
//   dL/du1_n = conj(E_n) I0
//   dL/dd1_n = Re[i theta'_n c_n conj(I0)] - sum_a G'_{n,a} Re[c_n conj(I_a)]
// with theta_n = k|x1|^2/(2 r0) + k d1 (sz - 1) = pi a (1 + q) + pi inc_d q/(1 + q)
// (at normal incidence the incident wave and the exp(-ik d1) of Eq. 5
// cancel; a tilted plane wave leaves its depth term, whose derivative is
// k (sz - 1) = pi inc_d / z0), theta' = pi a (1 + q)^2 / z0 + pi inc_d / z0 and
// G'_a = s_a (1 + q)^2 / z0, since
// dq/dd1 = z0 / (z0 - d1)^2 = (1 + q)^2 / z0.  These are the exact
// derivatives of the discrete forward computation, so <A x, y> = <x, A^H y>
// holds to rounding.
#include <algorithm>

#include "asfd_impl.cuh"
#include "fft.cuh"
#include "sample.cuh"

namespace asfd {

namespace {

struct InterpArgs {
    const float2* u1;
    const float* q;
    const AxisEntry* ax;
    const AxisEntry* ay;
    const AxisPos* px;
    const AxisPos* py;
    const float2* grid;   // b~ in storage coordinates, valid over the band
    float2* gu1;          // may be NULL
    float* gd1;           // may be NULL
    int n1x, n1y;
    int nfx, nfy;
    float half_w, beta_log2e, two_over_w, beta;
    float inv_z0;
    float inc_d;          // incident depth phase, half-turns per unit d1/z0
};

// psi and d psi / dz of the ES kernel for two taps at once (packed FP32x2; the
// MUFU square root and exponential).  CLAMP: taps that can reach the support's
// edge, 1 - u^2 floored at 1e-12 (the derivative is infinite there, where psi
// is e^-beta); other taps lie inside.  neg_c2 = -(2/w)^2;
// d psi/dz = psi z rsqrt(r) beta neg_c2.
template <bool CLAMP>
__device__ __forceinline__ void es_weight_deriv2_fast(float2 z, float neg_c2, float beta_log2e,
                                                      float beta_negc2, float2& psi, float2& dpsi)
{
    const float2 t = mul2(z, neg_c2);
    float2 r = fma2v(t, z, make_float2(1.f, 1.f));
    if constexpr (CLAMP) {
        r.x = fmaxf(r.x, 1e-12f);
        r.y = fmaxf(r.y, 1e-12f);
    }
    float2 rs, e;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(rs.x) : "f"(r.x));
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(rs.y) : "f"(r.y));
    const float2 s = fma2v(r, rs, make_float2(-1.f, -1.f));
    const float2 arg = mul2(s, beta_log2e);
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e.x) : "f"(arg.x));
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e.y) : "f"(arg.y));
    psi = e;
    dpsi = mul2(mul_f2(e, mul_f2(z, rs)), beta_negc2);
}

constexpr int kInterpWarps = 4;

// A sample per thread, 32 source columns x kInterpWarps rows of samples at a
// time, `iters` of them down the block.  A sample reads its W rows of cells as
// 16-byte pairs from the even column at or before its first tap (NX cells; the
// one or two that are no taps have zero weights): half the load instructions
// and L1 wavefronts of single cells, at constant offsets from one address per
// row.  Neighbouring samples' cells meet in L1 (86 % hits), so no window is
// kept: a register window of W x W cells, moved up row by row, left 8 warps per
// SM at 200 registers and took 603 us for 4096^2 samples, 34.5 for 1024^2; this
// takes 388 and 24.8.  Waits for the cells bound it, at half the issue slots;
// 8 warps per block 407, 16 (L1 overflows) 648, 2 warps 421; without the next
// sample's inputs loaded ahead 548.
// WRAP: footprints may wrap around the periodic grid.
template <int W, bool WRAP>
__global__ void __launch_bounds__(32 * kInterpWarps) interp_kernel(InterpArgs a, int iters)
{
    constexpr int NX = (W + 2) & ~1;
    chain_next();
    chain_wait();
    const int lane = threadIdx.x % 32, wid = threadIdx.x / 32;
    const int nx = blockIdx.x * 32 + lane;
    if (nx >= a.n1x) return;
    int ny = blockIdx.y * iters * kInterpWarps + wid;
    const int ny1 = min(a.n1y, (int)(blockIdx.y + 1) * iters * kInterpWarps);
    const int mx = a.nfx - 1, my = a.nfy - 1;
    const float neg_c2 = -a.two_over_w * a.two_over_w;
    const float beta_negc2 = a.beta * neg_c2;
    const AxisEntry ex = a.ax[nx];
    const AxisPos px = a.px[nx];
    // a sample's inputs, loaded one sample ahead
    float qn = 0.f;
    float2 un = make_float2(0.f, 0.f);
    AxisEntry eyn{};
    AxisPos pyn{};
    auto fetch = [&](int r) {
        if (r >= ny1) return;
        const size_t i = (size_t)r * a.n1x + nx;
        qn = __ldg(&a.q[i]);
        if (a.gd1) un = a.u1[i];
        eyn = a.ay[r];
        pyn = a.py[r];
    };
    fetch(ny);
    for (; ny < ny1; ny += kInterpWarps) {
        const size_t n = (size_t)ny * a.n1x + nx;
        const float q = qn;
        const float2 u = un;
        const AxisEntry ey = eyn;
        int l0x, l0y;
        float dx, dy;
        sample_pos(ex, ey, px, pyn, q, a.half_w, l0x, l0y, dx, dy);
        fetch(ny + kInterpWarps);
        const int odd = l0x & 1;
        int c0 = l0x - odd;
        if constexpr (!WRAP) {
            // (footprints lie inside the grid; clamped all the same)
            c0 = min(max(c0, 0), a.nfx - NX);
            l0y = min(max(l0y, 0), a.nfy - W);
        }
        // weights of window column j: tap j - odd
        float wx[NX], dwx[NX], wy[W + 1], dwy[W + 1];
        // (taps' offsets as (d + i) - w/2: the derivative is singular at the
        // support's edge, so its argument is rounded in one way everywhere)
        const float oddf = (float)odd;
#pragma unroll
        for (int j = 0; j < NX; j += 2) {
            float2 psi, dpsi;
            const float2 z = make_float2((dx + ((float)j - oddf)) - a.half_w,
                                         (dx + ((float)(j + 1) - oddf)) - a.half_w);
            if (j >= 2 && j + 3 < W)
                es_weight_deriv2_fast<false>(z, neg_c2, a.beta_log2e, beta_negc2, psi, dpsi);
            else
                es_weight_deriv2_fast<true>(z, neg_c2, a.beta_log2e, beta_negc2, psi, dpsi);
            // zero where column j (j + 1) is no tap
            const bool in0 = j > 0 ? (j < W || (j == W && odd)) : !odd;
            const bool in1 = j + 1 < W || (j + 1 == W && odd);
            wx[j] = in0 ? psi.x : 0.f;
            dwx[j] = in0 ? dpsi.x : 0.f;
            wx[j + 1] = in1 ? psi.y : 0.f;
            dwx[j + 1] = in1 ? dpsi.y : 0.f;
        }
#pragma unroll
        for (int b = 0; b < W; b += 2) {
            float2 psi, dpsi;
            const float2 z = make_float2((dy + (float)b) - a.half_w, (dy + (float)(b + 1)) - a.half_w);
            if (b >= 1 && b + 2 < W)
                es_weight_deriv2_fast<false>(z, neg_c2, a.beta_log2e, beta_negc2, psi, dpsi);
            else
                es_weight_deriv2_fast<true>(z, neg_c2, a.beta_log2e, beta_negc2, psi, dpsi);
            wy[b] = psi.x;
            dwy[b] = dpsi.x;
            wy[b + 1] = psi.y;
            dwy[b + 1] = dpsi.y;
        }
        float2 i0 = make_float2(0.f, 0.f), ixs = i0, iys = i0;
#pragma unroll
        for (int b = 0; b < W; ++b) {
            const int row = WRAP ? (l0y + b) & my : l0y + b;
            const float2* g = a.grid + (size_t)row * a.nfx;
            float2 s0 = make_float2(0.f, 0.f), sd = s0;
#pragma unroll
            for (int j = 0; j < NX; j += 2) {
                const float4 v = WRAP ? *reinterpret_cast<const float4*>(g + ((c0 + j) & mx))
                                      : reinterpret_cast<const float4*>(g + c0)[j / 2];
                const float2 v0 = make_float2(v.x, v.y), v1 = make_float2(v.z, v.w);
                s0 = fma2(v0, wx[j], s0);
                sd = fma2(v0, dwx[j], sd);
                s0 = fma2(v1, wx[j + 1], s0);
                sd = fma2(v1, dwx[j + 1], sd);
            }
            i0 = fma2(s0, wy[b], i0);
            ixs = fma2(sd, wy[b], ixs);
            iys = fma2(s0, dwy[b], iys);
        }
        // E = c / u1 (unit modulus prefactor)
        const float2 E = sample_value_fast(make_float2(1.f, 0.f), ex, ey, q, a.inc_d);
        if (a.gu1) a.gu1[n] = make_float2(E.x * i0.x + E.y * i0.y, E.x * i0.y - E.y * i0.x);
        if (a.gd1) {
            const float2 c = make_float2(u.x * E.x - u.y * E.y, u.x * E.y + u.y * E.x);
            const float opq = 1.0f + q;
            const float k2 = opq * opq * a.inv_z0;
            const float dtheta = 3.14159265358979f * ((ex.a + ey.a) * k2 + a.inc_d * a.inv_z0);
            const float gx = ex.s * k2, gy = ey.s * k2;
            // Re[i t c conj(I0)] = -t Im[c conj(I0)]
            const float im_c_i0 = c.y * i0.x - c.x * i0.y;
            const float re_c_ix = c.x * ixs.x + c.y * ixs.y;
            const float re_c_iy = c.x * iys.x + c.y * iys.y;
            a.gd1[n] = -dtheta * im_c_i0 - gx * re_c_ix - gy * re_c_iy;
        }
    }
}

}  // namespace

asfd_status launch_interp_grad(asfd_plan_s* P, const float2* u1, float2* gu1, float* gd1,
                               cudaStream_t st)
{
    InterpArgs a;
    a.u1 = u1;
    a.q = P->q;
    a.ax = P->ax;
    a.ay = P->ay;
    a.px = P->px;
    a.py = P->py;
    a.grid = P->grid;
    a.gu1 = gu1;
    a.gd1 = gd1;
    a.n1x = P->prm.n1x;
    a.n1y = P->prm.n1y;
    a.nfx = P->nfx;
    a.nfy = P->nfy;
    a.half_w = 0.5f * (float)P->w;
    a.beta_log2e = (float)(P->beta * 1.4426950408889634074);
    a.two_over_w = (float)(2.0 / P->w);
    a.beta = (float)P->beta;
    a.inv_z0 = (float)(1.0 / P->prm.z0);
    a.inc_d = (float)P->inc_d;
    // blocks of 32 columns x 4 iters rows: iters as large as leaves every SM
    // its resident blocks
    const int cols = (P->prm.n1x + 31) / 32;
    int iters = 16;
    while (iters > 1 &&
           (long long)cols * ((P->prm.n1y + iters * kInterpWarps - 1) / (iters * kInterpWarps)) < 2432)
        iters /= 2;
    const dim3 grid(cols, (P->prm.n1y + iters * kInterpWarps - 1) / (iters * kInterpWarps));
    cudaError_t e = cudaSuccess;
    switch (P->w) {
#define ASFD_IW(W)                                                                                    \
    case W:                                                                                           \
        e = P->wraps ? launch_chained(interp_kernel<W, true>, grid, 32 * kInterpWarps, 0, st, a, iters) \
                     : launch_chained(interp_kernel<W, false>, grid, 32 * kInterpWarps, 0, st, a, iters); \
        break;
        ASFD_IW(2) ASFD_IW(3) ASFD_IW(4) ASFD_IW(5) ASFD_IW(6) ASFD_IW(7) ASFD_IW(8) ASFD_IW(9)
        ASFD_IW(10) ASFD_IW(11) ASFD_IW(12) ASFD_IW(13) ASFD_IW(14) ASFD_IW(15) ASFD_IW(16)
#undef ASFD_IW
        default: return fail(ASFD_ERR_UNSUPPORTED, "kernel width outside 2..16");
    }
    if (e != cudaSuccess) return cuda_fail(e, "interp_kernel launch");
    return ASFD_OK;
}

}  // namespace asfd
