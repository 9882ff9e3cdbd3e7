// One-dimensional form with explicit source samples (an extension: the
// paper's own experiments, Sec. 3, are line sources sampled along their arc
// length).  Sample j sits at x1[j] with height d1[j] and quadrature weight
// w[j] (its extent along x1); the destination line is x2 = (m - M/2) p2.
// Eq. 7 in one dimension, with r0 = z0 - d1 and the incident plane wave
// u_I = exp(ik(s x1 + sz d1)), sz = sqrt(1 - s^2):
//
//   u2(x2) = exp(ik(z0 + x2^2/(2 z0))) / sqrt(i lambda z0)
//            * sum_j w u_I u1 exp(ik(-d1 + x1^2/(2 r0))) exp(-ik x1 x2 / r0)
//
// (the 1D Fresnel prefactor 1/sqrt(i lambda z0) is a reading; the paper
// prints the 2D forms).  As in 2D this is a type-1 NUFFT at the fine-grid
// coordinate g = x1 p2 nf/(lambda r0): the plan forms, in FP64 and once, each
// sample's prefactor E_j = w exp(i pi h), h = x1^2/(lambda r0) +
// 2 (s x1 + (sz - 1) d1)/lambda half-turns reduced modulo 2, and the
// integer/fraction split of g + nf/2; an execution multiplies u1 by E,
// spreads with the ES kernel (float2 atomic adds into the nf-point line),
// transforms the line with the library's Stockham FFT and applies
// (-1)^m' exp(ik x2^2/(2 z0)) / psi_hat(2 pi m'/nf) and the global factor:
// one kernel of one block up to kLineOneBlock samples, with a spread kernel
// before it above.  Such a line is all latency: as a memset and three kernels
// 1024 samples took 6.7 us of GPU time in 21.
#include <algorithm>
#include <cmath>
#include <mutex>
#include <new>
#include <string>
#include <vector>

#include "asfd_impl.cuh"
#include "fft.cuh"
#include "sample.cuh"

struct asfd_line_plan_s {
    asfd_line_params prm;
    int device = 0;
    int n = 0, nf = 0, w = 0;
    double beta = 0.0;
    float2* e = nullptr;      // [n] per-sample prefactor (with the weight)
    int* bi = nullptr;        // [n] integer part of g + nf/2 (mod nf)
    float* bf = nullptr;      // [n] fraction
    float2* grid = nullptr;   // [nf], zero between calls
    bool clean = false;       // the grid is zero
    const float2* tw = nullptr;  // twiddles of nf points (a process-wide table)
    float2* c = nullptr;      // [m2] destination table
    double* quad = nullptr;
    unsigned* status = nullptr;
};

namespace asfd {

namespace {

__device__ __forceinline__ double line_reduce(double h) { return h - 2.0 * rint(0.5 * h); }

__global__ void line_prep_kernel(const double* __restrict__ x1, const double* __restrict__ d1,
                                 const double* __restrict__ w, int n, double lambda, double z0,
                                 double p2, int nf, double s, double sz, float2* __restrict__ e,
                                 int* __restrict__ bi, float* __restrict__ bf,
                                 unsigned* __restrict__ status)
{
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= n) return;
    const double x = x1[j], h = d1[j], wt = w[j];
    if (!isfinite(x) || !isfinite(h) || !isfinite(wt) || !(h < z0)) {
        atomicOr(status, kStatusBadD1);
        e[j] = make_float2(0.f, 0.f);
        bi[j] = 0;
        bf[j] = 0.f;
        return;
    }
    const double r0 = z0 - h;
    const double ph = line_reduce(x * x / (lambda * r0)) + line_reduce(2.0 * (s * x + (sz - 1.0) * h) / lambda);
    double sn, cs;
    sincospi(ph, &sn, &cs);
    e[j] = make_float2((float)(wt * cs), (float)(wt * sn));
    const double g = x * p2 * (double)nf / (lambda * r0) + 0.5 * (double)nf;
    const double gr = g - (double)nf * floor(g / (double)nf);
    int b = (int)floor(gr);
    double f = gr - (double)b;
    if (b >= nf) b -= nf;
    bi[j] = b;
    bf[j] = (float)f;
}

// C[k] = (-1)^m' exp(i pi x2^2/(lambda z0)) / psi_hat(2 pi m'/nf) * exp(ik z0) exp(-i pi/4)
//        / sqrt(lambda z0),  m' = k - m2/2
__global__ void line_dest_kernel(float2* __restrict__ C, int m2, double p2, double lambda,
                                 double z0, int nf, const double* __restrict__ quad, int nq)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= m2) return;
    const int mp = k - m2 / 2;
    const double x2 = (double)mp * p2;
    double psi_hat = 0.0;
    for (int i = 0; i < nq; ++i) psi_hat += quad[nq + i] * cospi(2.0 * (double)mp * quad[i] / (double)nf);
    psi_hat *= 2.0;
    const double ph = line_reduce(x2 * x2 / (lambda * z0)) + line_reduce(2.0 * z0 / lambda) - 0.25;
    double sn, cs;
    sincospi(ph, &sn, &cs);
    const double a = ((mp & 1) ? -1.0 : 1.0) / (psi_hat * sqrt(lambda * z0));
    C[k] = make_float2((float)(a * cs), (float)(a * sn));
}

struct LineArgs {
    const float2* u1;
    const float2* e;
    const int* bi;
    const float* bf;
    int n, nf, w;
    float half_w, two_over_w, beta_log2e;
    float2* grid;
    const float2* C;
    int m2;
    float2* u2;
    const float2* tw;
};

// Samples that the transform's own block spreads: as many as it has threads, and
// at most two per fine cell (their atomic adds meet in few cells).  At 1024
// destination points 7.2 us a call against 9.9 with a kernel for the spread
// (1024 samples), even at 2048 samples, 24.1 against 9.8 at 8192; at 128 points
// 8.3 against 10.9 (512 samples), 11.7 against 9.7 (1024).
constexpr int kLineOneBlock = 1024;

// Adds sample j's taps to the line (periodic).
__device__ __forceinline__ void line_spread_sample(const LineArgs& a, int j)
{
    const float2 u = a.u1[j], ej = __ldg(&a.e[j]);
    const float2 c = make_float2(u.x * ej.x - u.y * ej.y, u.x * ej.y + u.y * ej.x);
    const float f = __ldg(&a.bf[j]) - a.half_w;
    const float cf = ceilf(f);
    const int l0 = __ldg(&a.bi[j]) + (int)cf;
    const float dx = cf - f;
    const int mask = a.nf - 1;
#pragma unroll 4
    for (int i = 0; i < a.w; ++i) {
        const float wv = es_weight_fast(dx + (float)i - a.half_w, a.two_over_w, a.beta_log2e);
        atomicAdd(&a.grid[(l0 + i) & mask], make_float2(c.x * wv, c.y * wv));
    }
}

__global__ void __launch_bounds__(256) line_spread_kernel(LineArgs a)
{
    chain_next();
    chain_wait();
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j < a.n) line_spread_sample(a, j);
}

// Threads of the transform's block, at most: as many as there are samples to
// spread, or as transform the line; 512 for 8192 points, whose 32 values per
// thread fit the 128 registers that leaves (64 of a block of 1024: 324 bytes of
// spills).
template <int L, bool SPREAD>
__host__ __device__ constexpr int line_threads()
{
    constexpr int tpl = FftShape<L>::TPL < 32 ? 32 : FftShape<L>::TPL;
    return !SPREAD ? tpl : L == 8192 ? 512 : 1024;
}

// The block spreads the samples (SPREAD), and its first TPL threads transform
// the line, leave it zero for the next call and write the destination.
template <int L, bool SPREAD>
__global__ void __launch_bounds__(line_threads<L, SPREAD>()) line_transform_kernel(LineArgs a)
{
    extern __shared__ float2 sm[];
    chain_next();
    chain_wait();
    const int t = threadIdx.x;
    if constexpr (SPREAD) {
        for (int j = t; j < a.n; j += blockDim.x) line_spread_sample(a, j);
        __threadfence();  // the sums are in L2, where the loads below read
        __syncthreads();
    }
    if (t >= FftShape<L>::TPL) return;
    auto ld = [&](int i) -> float2 {
        const float2 v = __ldcg(&a.grid[i]);
        a.grid[i] = make_float2(0.f, 0.f);
        return v;
    };
    const int half = a.m2 / 2;
    auto st = [&](int i, float2 v) {
        int k;
        if (i < half) k = i + half;
        else if (i >= L - half) k = i - (L - half);
        else return;
        a.u2[k] = cmul(v, __ldg(&a.C[k]));
    };
    fft_line<L, -1>(t, sm, a.tw, ld, st);
}

template <int L>
cudaError_t line_launch(const LineArgs& a, bool spread, cudaStream_t st)
{
    constexpr size_t smem = sizeof(float2) * FftShape<L>::SMEM;
    constexpr int TPL = FftShape<L>::TPL;
    if constexpr (smem > 48 * 1024) {
        static std::once_flag once;
        static cudaError_t attr = cudaSuccess;
        std::call_once(once, [] {
            attr = cudaFuncSetAttribute(line_transform_kernel<L, true>,
                                        cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
            if (attr == cudaSuccess)
                attr = cudaFuncSetAttribute(line_transform_kernel<L, false>,
                                            cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        });
        if (attr != cudaSuccess) return attr;
    }
    if (!spread)
        return launch_chained(line_transform_kernel<L, false>, dim3(1), line_threads<L, false>(), smem,
                              st, a);
    int threads = std::min(line_threads<L, true>(), (a.n + 31) / 32 * 32);
    threads = std::max(threads, std::max(32, TPL));
    return launch_chained(line_transform_kernel<L, true>, dim3(1), (unsigned)threads, smem, st, a);
}

void line_free(asfd_line_plan_s* P)
{
    void* bufs[] = {P->e, P->bi, P->bf, P->grid, P->c, P->quad, P->status};
    for (void* b : bufs)
        if (b) cudaFree(b);
    delete P;
}

}  // namespace
}  // namespace asfd

using namespace asfd;

extern "C" {

asfd_status asfd_line_plan_create(asfd_line_plan* out, const asfd_line_params* p,
                                  const double* x1_dev, const double* d1_dev, const double* w_dev,
                                  int n, void* stream)
{
    clear_error();
    if (!out || !p || !x1_dev || !d1_dev || !w_dev || n < 1)
        return fail(ASFD_ERR_ARG, "out, params and sample arrays must be non-NULL, n >= 1");
    *out = nullptr;
    if (p->m2 < 2 || p->m2 % 2) return fail(ASFD_ERR_ARG, "m2 must be even and >= 2");
    const double pos[] = {p->p2, p->lambda, p->z0, p->sigma};
    for (double v : pos)
        if (!(std::isfinite(v) && v > 0.0))
            return fail(ASFD_ERR_ARG, "p2, wavelength, z0 and sigma must be finite and > 0");
    if (!(std::isfinite(p->incidence_s) && p->incidence_s * p->incidence_s < 1.0))
        return fail(ASFD_ERR_ARG, "incidence direction cosine needs s^2 < 1");
    if (p->kernel_width < 2 || p->kernel_width > 16)
        return fail(ASFD_ERR_UNSUPPORTED, "kernel_width must be in [2, 16]");
    const double fnf = p->sigma * p->m2;
    const int nf = (int)std::lround(fnf);
    if (std::fabs(fnf - nf) > 1e-9 * fnf || nf < 64 || nf > 16384 || (nf & (nf - 1)))
        return fail(ASFD_ERR_UNSUPPORTED, "sigma*m2 must be a power of two in [64, 16384]");
    if (p->kernel_width >= nf / 2) return fail(ASFD_ERR_UNSUPPORTED, "kernel wider than half the line");
    if (!(std::isfinite(p->es_beta) && p->es_beta >= 0.0))
        return fail(ASFD_ERR_ARG, "es_beta must be finite and >= 0");
    asfd_line_plan_s* P = new (std::nothrow) asfd_line_plan_s();
    if (!P) return fail(ASFD_ERR_NOMEM, "host allocation of the plan failed");
    P->prm = *p;
    P->n = n;
    P->nf = nf;
    P->w = p->kernel_width;
    const double pi = 3.14159265358979323846;
    P->beta = p->es_beta > 0.0 ? p->es_beta
                               : (p->sigma == 2.0 ? 2.30 * p->kernel_width
                                                  : 0.97 * pi * (1.0 - 1.0 / (2.0 * p->sigma)) *
                                                        p->kernel_width);
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    asfd_status s = [&]() -> asfd_status {
        ASFD_CUDA(cudaGetDevice(&P->device));
        ASFD_CUDA(cudaMalloc(&P->e, sizeof(float2) * n));
        ASFD_CUDA(cudaMalloc(&P->bi, sizeof(int) * n));
        ASFD_CUDA(cudaMalloc(&P->bf, sizeof(float) * n));
        ASFD_CUDA(cudaMalloc(&P->grid, sizeof(float2) * nf));
        ASFD_CUDA(cudaMalloc(&P->c, sizeof(float2) * p->m2));
        ASFD_CUDA(cudaMalloc(&P->status, sizeof(unsigned)));
        std::vector<double> h;
        const int nq = es_quadrature(P->w, P->beta, h);
        ASFD_CUDA(cudaMalloc(&P->quad, sizeof(double) * h.size()));
        ASFD_CUDA(cudaMemcpyAsync(P->quad, h.data(), sizeof(double) * h.size(),
                                  cudaMemcpyHostToDevice, st));
        ASFD_CUDA(cudaMemsetAsync(P->status, 0, sizeof(unsigned), st));
        ASFD_CUDA(cudaMemsetAsync(P->grid, 0, sizeof(float2) * nf, st));
        const asfd_status ts = fft_line_twiddles(nf, &P->tw, st);
        if (ts != ASFD_OK) return ts;
        const double sz = std::sqrt(1.0 - p->incidence_s * p->incidence_s);
        line_prep_kernel<<<(n + 255) / 256, 256, 0, st>>>(x1_dev, d1_dev, w_dev, n, p->lambda,
                                                           p->z0, p->p2, nf, p->incidence_s, sz,
                                                           P->e, P->bi, P->bf, P->status);
        line_dest_kernel<<<(p->m2 + 255) / 256, 256, 0, st>>>(P->c, p->m2, p->p2, p->lambda,
                                                               p->z0, nf, P->quad, nq);
        ASFD_CUDA(cudaGetLastError());
        unsigned bad = 0;
        ASFD_CUDA(cudaMemcpyAsync(&bad, P->status, sizeof(unsigned), cudaMemcpyDeviceToHost, st));
        ASFD_CUDA(cudaStreamSynchronize(st));
        if (bad)
            return fail(ASFD_ERR_ARG, "x1, d1 and w must be finite and every d1 below z0");
        P->clean = true;
        return ASFD_OK;
    }();
    if (s != ASFD_OK) {
        const std::string msg = asfd_last_error();
        line_free(P);
        return fail(s, msg);
    }
    *out = P;
    return ASFD_OK;
}

asfd_status asfd_line_execute(asfd_line_plan P, const float* u1_dev, float* u2_dev, void* stream)
{
    clear_error();
    if (!P || !u1_dev || !u2_dev) return fail(ASFD_ERR_ARG, "NULL argument");
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    int dev = -1;
    cudaGetDevice(&dev);
    if (dev != P->device) {
        const cudaError_t e = cudaSetDevice(P->device);
        if (e != cudaSuccess) return cuda_fail(e, "cudaSetDevice");
    }
    asfd_status s = [&]() -> asfd_status {
        LineArgs a;
        a.u1 = reinterpret_cast<const float2*>(u1_dev);
        a.e = P->e;
        a.bi = P->bi;
        a.bf = P->bf;
        a.n = P->n;
        a.nf = P->nf;
        a.w = P->w;
        a.half_w = 0.5f * (float)P->w;
        a.two_over_w = (float)(2.0 / P->w);
        a.beta_log2e = (float)(P->beta * 1.4426950408889634074);
        a.grid = P->grid;
        a.C = P->c;
        a.m2 = P->prm.m2;
        a.u2 = reinterpret_cast<float2*>(u2_dev);
        a.tw = P->tw;
        // (the transform leaves the line zero; not so after a failed launch)
        if (!P->clean) ASFD_CUDA(cudaMemsetAsync(P->grid, 0, sizeof(float2) * P->nf, st));
        P->clean = false;
        const bool one = P->n <= std::min(kLineOneBlock, 2 * P->nf);
        if (!one) ASFD_CUDA(launch_chained(line_spread_kernel, dim3((P->n + 255) / 256), 256, 0, st, a));
        cudaError_t e = cudaErrorInvalidValue;
        switch (P->nf) {
#define ASFD_LT(L) case L: e = line_launch<L>(a, one, st); break;
            ASFD_LT(64) ASFD_LT(128) ASFD_LT(256) ASFD_LT(512) ASFD_LT(1024) ASFD_LT(2048) ASFD_LT(4096)
            ASFD_LT(8192) ASFD_LT(16384)
#undef ASFD_LT
            default: break;
        }
        if (e != cudaSuccess) return cuda_fail(e, "line_transform_kernel launch");
        P->clean = true;
        return ASFD_OK;
    }();
    if (dev != P->device && dev >= 0) cudaSetDevice(dev);
    return s;
}

asfd_status asfd_line_destroy(asfd_line_plan P)
{
    clear_error();
    if (!P) return ASFD_OK;
    int dev = -1;
    cudaGetDevice(&dev);
    const int own = P->device;  // P is gone after line_free
    if (dev != own) cudaSetDevice(own);
    line_free(P);
    if (dev != own && dev >= 0) cudaSetDevice(dev);
    return ASFD_OK;
}

}  // extern "C"
