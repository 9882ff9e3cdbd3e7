// Direct (O(N^2 M^2)) evaluation of the diffraction sums at destination
// points, on the GPU: Eq. 7 (the Fourier form the NUFFT computes), Eq. 5 (the
// destination chirp with r0 = z0 - d1 per sample, before the approximation of
// Eq. 6) and Eq. 2 (the Huygens sum with the exact distance of Eq. 3, before
// the Fresnel expansion of Eq. 4).  They measure what those approximations
// cost at 2D scale and serve as a fast reference on sampled points.
//
// The phase of a pair is formed modulo one turn in 64-bit fixed point.  At a
// destination index j = m - M/2 the phases of Eqs. 5 and 7 are, in turns,
//   Eq. 7: A - B jx - C jy
//          A = |x1|^2/(2 lambda r0) + (s.x1 + (sz - 1) d1)/lambda (the last
//          term is u_I exp(-ik d1) for a plane wave with direction cosines
//          (sx, sy, sz); zero at normal incidence), B = x1 p2x/(lambda r0),
//          C = y1 p2y/(lambda r0)
//   Eq. 5: the same + D R, D = p2x^2/(2 lambda r0), R = jx^2 + (p2y/p2x)^2 jy^2,
//          an integer for equal pitches (else D R is formed in FP64)
// The per-sample A, B, C, D are formed in FP64 and reduced modulo 1 there, to
// 2^-50 turns (D, which is small, to 2^-64); products with the integer
// indices and their sum are then exact modulo 2^64, which is the reduction
// modulo one turn.  (With FP64 arithmetic per pair -- 2 lanes per clock and
// SM, where integer multiply-adds have 64 -- and one block per point group 256
// points of 1024^2 samples took 28.6 ms; now 0.46 ms, at an error against 64
// bits of 5e-8 instead of 6e-8.)
//   Eq. 2: 2 (s.x1 + sz d1 + r)/lambda half-turns, amplitude 1/r^2,
//          r = |(x2 - x1, z0 - d1)|, in FP64 from an FP32 reciprocal square
//          root and its residual to third order (as good as an FP64 square
//          root, which is slow here: r counts up to 1e8 half-turns and more).
// The high 32 bits of the phase go to an FP32 sine and cosine on a quarter
// turn (polynomials, |error| < 6e-8); products with u1 are FP32 and the sums
// of a thread are carried as an FP32 value and its exact rounding errors
// (two-sum), which meet in FP64.
// Outer factors: p1x p1y exp(ik(z0 + |x2|^2/(2 z0)))/(i lambda z0) (Eq. 7),
// p1x p1y exp(ik z0)/(i lambda z0) (Eq. 5), p1x p1y z0/(i lambda) (Eq. 2).
#include <algorithm>
#include <cmath>
#include <string>
#include <type_traits>

#include "asfd_impl.cuh"
#include "fft.cuh"

namespace asfd {

namespace {

constexpr int kDirectThreads = 256;
constexpr int kDirectPoints = 8;      // destination points per block (shares the sample loads)
constexpr int kDirectBlocks = 4;      // blocks per SM that the samples are split into
constexpr int kDirectMaxRows = 1024;  // samples per thread, at most (of one two-sum)

struct DirectGeom {
    int n1x, n1y, m2x, m2y;
    double p1x, p1y, p2x, p2y, lambda, z0;
    double sx, sy, sz;  // incident plane wave direction cosines
    double ox, oy;      // source grid offset
    double inv_lambda;
};

// What direct_sum_kernel evaluates: the paper's equations, and Eq. 5 for
// destination pitches that differ (kEq5Uneven).
enum DirectForm { kEq2 = 2, kEq5 = 5, kEq5Uneven = 6, kEq7 = 7 };

// Per-sample terms, 32-byte aligned.  Eq. 5/7: {A', -B, -C, D} as 64-bit
// fractions of a turn (A' = A at the index origin below; D as a double for
// uneven pitches); Eq. 2: the doubles {x1x, x1y, (z0 - d1)^2,
// 2 (s.x1 + sz d1)/lambda mod 2}
struct alignas(32) DirectTerms {
    unsigned long long a, b, c, d;
};

// fractional part of v (turns) in units of 2^-64, to 2^-50: after the
// reduction to [-1/2, 1/2] the sum with 1.5 2^2 has an ulp of 2^-50
__device__ __forceinline__ unsigned long long turn_fraction(double v)
{
    const double f = v - rint(v);
    return (unsigned long long)__double_as_longlong(f + 6.0) << 14;
}

// Indices enter the products as unsigned 32-bit numbers m + 2^31 (any int is
// allowed); A' moves the origin there, exactly modulo one turn.
constexpr unsigned kIndexBias = 0x80000000u;

// A block takes 256 columns x kPrepRows rows: a thread's column terms serve its
// rows, the rows' terms are formed once per block (FP64 is 2 lanes per clock
// and SM: 45 FP64 operations per sample in a thread each took 90 us at 1024^2).
// *bad is set when a height or a term of the phase is not finite (d1 is not
// checked: a NaN or an infinity, d1 = z0, or a term that overflows makes every
// sum a NaN, which fixed point cannot carry).
constexpr int kPrepRows = 8;

// by the bits: FP64 comparisons are slow here
__device__ __forceinline__ bool not_finite(double v)
{
    return (__double2hiint(v) & 0x7ff00000) == 0x7ff00000;
}

__global__ void __launch_bounds__(256)
direct_prep_kernel(DirectGeom g, const double* d1, int form, DirectTerms* out, unsigned* bad)
{
    __shared__ double ys[kPrepRows];
    chain_next();
    chain_wait();
    const int nx = blockIdx.x * 256 + threadIdx.x, ny0 = blockIdx.y * kPrepRows;
    if (threadIdx.x < kPrepRows)
        ys[threadIdx.x] = (ny0 + (int)threadIdx.x - g.n1y / 2) * g.p1y + g.oy;
    __syncthreads();
    if (nx >= g.n1x) return;
    const double x = (nx - g.n1x / 2) * g.p1x + g.ox;
    const double xx = x * x, xp = x * g.p2x, half_pp = 0.5 * g.p2x * g.p2x;
    const bool tilted = g.sx != 0.0 || g.sy != 0.0;
    const int rows = min(kPrepRows, g.n1y - ny0);
    for (int r = 0; r < rows; ++r) {
        const size_t n = (size_t)(ny0 + r) * g.n1x + nx;
        const double y = ys[r], h = d1[n];
        DirectTerms t;
        if (form == kEq2) {
            const double z = g.z0 - h;
            const double w = 2.0 * (g.sx * x + g.sy * y + g.sz * h) * g.inv_lambda;
            t.a = (unsigned long long)__double_as_longlong(x);
            t.b = (unsigned long long)__double_as_longlong(y);
            t.c = (unsigned long long)__double_as_longlong(z * z);
            t.d = (unsigned long long)__double_as_longlong(w - 2.0 * rint(0.5 * w));
        } else {
            const double inv = 1.0 / (g.lambda * (g.z0 - h));
            const double ta = 0.5 * (xx + y * y) * inv, tb = xp * inv, tc = y * g.p2y * inv;
            const unsigned long long b = turn_fraction(tb);
            const unsigned long long c = turn_fraction(tc);
            t.a = turn_fraction(ta) + b * ((unsigned long long)kIndexBias + (unsigned)(g.m2x / 2)) +
                  c * ((unsigned long long)kIndexBias + (unsigned)(g.m2y / 2));
            // (1 / (lambda (z0 - h)) of an infinite height is a finite zero)
            bool nonfinite = not_finite(h) || not_finite(ta) || not_finite(tb) || not_finite(tc);
            if (tilted) {
                const double ti = (g.sx * x + g.sy * y + (g.sz - 1.0) * h) * g.inv_lambda;
                t.a += turn_fraction(ti);
                nonfinite = nonfinite || not_finite(ti);
            }
            t.b = 0ull - b;
            t.c = 0ull - c;
            const double d = half_pp * inv;
            t.d = 0;
            if (form == kEq5Uneven)
                t.d = (unsigned long long)__double_as_longlong(d);
            else if (form == kEq5)
                t.d = (unsigned long long)__double2ll_rn((d - rint(d)) * 18446744073709551616.0);
            if (nonfinite || not_finite(d)) atomicOr(bad, 1u);
        }
        out[n] = t;
    }
}

// cos and sin of two phases p 2^-32 turns.  The nearest quarter turn is the
// top two bits of p + 2^29, the rest is x = (p << 2) 2^-32 quarter turns in
// [-1/2, 1/2): there sin(pi x/2) = x S(x^2) and cos(pi x/2) = 1 + x^2 C(x^2),
// with S and C interpolated at the Chebyshev nodes of x^2 in [0, 1/4] (degree
// 3); the leading coefficient of S, pi/2, is split in two so that its own
// rounding does not show (rms error 2.4e-8 of a unit vector; 2.1e-8 is the
// rounding to FP32 alone).  Two points at a time: the polynomials run in
// packed FP32x2, the choice of the quadrant on the integer pipe.  (Half
// turns, with longer polynomials and one sign to choose, are no faster and
// less exact, 3.7e-8: x^2 of a larger x is rounded.)
__device__ __forceinline__ float2 pair2(float v) { return make_float2(v, v); }

__device__ __forceinline__ void to_quadrant(unsigned p, float s, float c, float& sn, float& cs)
{
    const unsigned t = p + 0x20000000u;
    const bool odd = (t & 0x40000000u) != 0;
    const unsigned c0 = __float_as_uint(odd ? s : c), s0 = __float_as_uint(odd ? c : s);
    cs = __uint_as_float(c0 ^ ((t ^ (t << 1)) & 0x80000000u));
    sn = __uint_as_float(s0 ^ (t & 0x80000000u));
}

__device__ __forceinline__ void turn_sincos2(unsigned p0, unsigned p1, float2& sn, float2& cs)
{
    const float2 x = mul_f2(make_float2((float)(int)(p0 << 2), (float)(int)(p1 << 2)),
                            pair2(2.3283064365386963e-10f));
    const float2 y = mul_f2(x, x);
    float2 s = fma_f2(y, pair2(-0.004602149f), pair2(0.07968022f));
    s = fma_f2(y, s, pair2(-0.6459635f));
    s = fma_f2(y, s, pair2(-4.371139e-8f));  // pi/2 - 1.5707964f
    s = fma_f2(x, pair2(1.5707964f), mul_f2(x, s));
    float2 c = fma_f2(y, pair2(0.0009067399f), pair2(-0.020861529f));
    c = fma_f2(y, c, pair2(0.2536694f));
    c = fma_f2(y, c, pair2(-1.2337005f));
    c = fma_f2(y, c, pair2(1.0f));
    to_quadrant(p0, s.x, c.x, sn.x, cs.x);
    to_quadrant(p1, s.y, c.y, sn.y, cs.y);
}

// sum += v on a pair, with the low part of the sum in -low (Kahan)
__device__ __forceinline__ void kahan_add(float2& sum, float2& low, float2 v)
{
    const float2 y = csub(v, low);
    const float2 t = cadd(sum, y);
    low = csub(csub(t, sum), y);
    sum = t;
}

// Resident blocks per SM (three need Eq. 7's 80 registers)
__host__ __device__ constexpr int direct_blocks_per_sm(int form)
{
    return form == kEq7 ? 3 : 2;
}

// Point groups in x, sample chunks in y: the chunk's sums over its samples of
// kDirectPoints points, to part[chunk][point].  Bound by the FMA pipe and
// instruction issue together (60 and 55 % busy: 12 packed operations, 4
// integer multiply-adds and 10 integer operations a pair), so more resident
// warps, a sample's loads one iteration ahead and one exact wave of blocks
// made no difference (0.39-0.42 ms against 0.385 ms at 256 points of 1024^2
// samples).  One block per group alone leaves 120 of the 152 SMs idle there,
// so the samples are split as well.
template <DirectForm FORM>
__global__ void __launch_bounds__(kDirectThreads, direct_blocks_per_sm(FORM))
direct_sum_kernel(DirectGeom g, const DirectTerms* s, const float2* u1, int npts, const int* mx,
                  const int* my, size_t chunk, double2* part)
{
    constexpr int P = kDirectPoints;
    static_assert(P % 2 == 0 && P <= 32, "points in pairs, a lane each for the sums");
    chain_next();
    chain_wait();
    __shared__ double red[2][P][kDirectThreads / 32];
    const int p0 = blockIdx.x * P;
    unsigned ix[P], iy[P];
    double x2x[P], x2y[P];
    unsigned long long r5[P];  // Eq. 5's R
    double r5u[P];
#pragma unroll
    for (int j = 0; j < P; ++j) {
        const int i = min(p0 + j, npts - 1);
        const int jx = mx[i], jy = my[i];
        ix[j] = (unsigned)jx + kIndexBias;
        iy[j] = (unsigned)jy + kIndexBias;
        if constexpr (FORM == kEq2) {
            x2x[j] = ((double)jx - g.m2x / 2) * g.p2x;
            x2y[j] = ((double)jy - g.m2y / 2) * g.p2y;
        }
        if constexpr (FORM == kEq5) {
            const long long kx = (long long)jx - g.m2x / 2, ky = (long long)jy - g.m2y / 2;
            r5[j] = (unsigned long long)kx * (unsigned long long)kx +
                    (unsigned long long)ky * (unsigned long long)ky;
        }
        if constexpr (FORM == kEq5Uneven) {
            const double kx = (double)jx - g.m2x / 2;
            const double ky = ((double)jy - g.m2y / 2) * (g.p2y / g.p2x);
            r5u[j] = kx * kx + ky * ky;
        }
    }
    // phase (2^-32 turns) and amplitude of the sample's terms t at point j
    // (exact: with FP64 square root and reciprocal, for a thread's second pass)
    auto phase = [&](auto exact, const ulonglong2& t0, const ulonglong2& t1, int j, float& amp) -> unsigned {
        if constexpr (FORM == kEq2) {
            const double dx = x2x[j] - __longlong_as_double((long long)t0.x);
            const double dy = x2y[j] - __longlong_as_double((long long)t0.y);
            const double r2 = fma(dx, dx, fma(dy, dy, __longlong_as_double((long long)t1.x)));
            double r;
            if constexpr (exact.value) {
                r = sqrt(r2);
                amp = (float)(1.0 / r2);
            } else {
                const float r2f = (float)r2;
                // with y = (1 + e)/r: ra = r2 y = r (1 + e), the residual r2 - ra^2 =
                // -(2e + e^2) r2, and r = ra + c + (3/4) t c up to e^3, with c =
                // residual y/2 and t = residual y^2 = -2e, for which FP32 is enough
                const float y = rsqrtf(r2f);
                const double yd = (double)y, ra = r2 * yd, res = fma(-ra, ra, r2);
                const double c = 0.5 * yd * res;
                const float t = y * ((float)res * y);
                r = ra + fma(c, (double)(0.75f * t), c);
                // 1/r^2 = y^2 (1 + t) up to t^2, y^2 with its rounding error
                const float a0 = y * y;
                amp = a0 + fmaf(a0, t, fmaf(y, y, -a0));
                // (out of FP32's range: a NaN sends the thread to its second pass)
                if (!(r2f > 1e-24f && r2f < 1e30f)) amp = __int_as_float(0x7fc00000);
            }
            double h = fma(2.0 * g.inv_lambda, r, __longlong_as_double((long long)t1.y));
            h -= 2.0 * rint(0.5 * h);
            if constexpr (exact.value)
                if (!isfinite(h)) amp = __int_as_float(0x7fc00000);  // (no such phase)
            // units of 2^-31 half-turns from the low bits of h + 1.5 2^21
            return (unsigned)__double_as_longlong(h + 3145728.0);
        } else {
            unsigned long long ph = t0.x + t0.y * (unsigned long long)ix[j] +
                                    t1.x * (unsigned long long)iy[j];
            if constexpr (FORM == kEq5) ph += t1.y * r5[j];
            if constexpr (FORM == kEq5Uneven)
                ph += turn_fraction(__longlong_as_double((long long)t1.y) * r5u[j]);
            return (unsigned)(ph >> 32);
        }
    };
    // products u exp(2 pi i phase) amp of points j and j + 1
    auto products = [&](auto exact, const ulonglong2& t0, const ulonglong2& t1, float2 u, int j,
                        float2& re, float2& im) {
        float2 amp = pair2(1.f), sn, cs;
        const unsigned pa = phase(exact, t0, t1, j, amp.x), pb = phase(exact, t0, t1, j + 1, amp.y);
        turn_sincos2(pa, pb, sn, cs);
        float2 ux = pair2(u.x), uy = pair2(u.y);
        if constexpr (FORM == kEq2) {
            ux = mul_f2(ux, amp);
            uy = mul_f2(uy, amp);
        }
        re = fma_f2(cs, ux, mul_f2(sn, make_float2(-uy.x, -uy.y)));
        im = fma_f2(cs, uy, mul_f2(sn, ux));
    };
    const size_t total = (size_t)g.n1x * g.n1y;
    const size_t beg = blockIdx.y * chunk, end = min(total, beg + chunk);
    const int lane = threadIdx.x % 32, warp = threadIdx.x / 32;
    if (lane < P) red[0][lane][warp] = red[1][lane][warp] = 0.0;
    __syncwarp();
    // at most kDirectMaxRows samples of a thread in one compensated sum
    for (size_t b0 = beg; b0 < end; b0 += (size_t)kDirectMaxRows * kDirectThreads) {
        const size_t b1 = min(end, b0 + (size_t)kDirectMaxRows * kDirectThreads);
        float2 sr[P / 2], lr[P / 2], si[P / 2], li[P / 2];  // of points 2k and 2k + 1
#pragma unroll
        for (int k = 0; k < P / 2; ++k) sr[k] = lr[k] = si[k] = li[k] = pair2(0.f);
        for (size_t n = b0 + threadIdx.x; n < b1; n += kDirectThreads) {
            const ulonglong2* tp = reinterpret_cast<const ulonglong2*>(s + n);
            const ulonglong2 t0 = tp[0], t1 = tp[1];
            const float2 u = u1[n];
#pragma unroll
            for (int k = 0; k < P / 2; ++k) {
                float2 re, im;
                products(std::false_type{}, t0, t1, u, 2 * k, re, im);
                kahan_add(sr[k], lr[k], re);
                kahan_add(si[k], li[k], im);
            }
        }
        double vs[2 * P];  // re and im of each point
#pragma unroll
        for (int k = 0; k < P / 2; ++k) {
            double v[4] = {(double)sr[k].x - lr[k].x, (double)si[k].x - li[k].x,
                           (double)sr[k].y - lr[k].y, (double)si[k].y - li[k].y};
            // overflow of an FP32 sum, infinite fields, distances out of FP32's
            // range: the sums in FP64
            if (!(isfinite(v[0]) && isfinite(v[1]) && isfinite(v[2]) && isfinite(v[3]))) {
                v[0] = v[1] = v[2] = v[3] = 0.0;
                for (size_t n = b0 + threadIdx.x; n < b1; n += kDirectThreads) {
                    const ulonglong2* tp = reinterpret_cast<const ulonglong2*>(s + n);
                    float2 re, im;
                    products(std::true_type{}, tp[0], tp[1], u1[n], 2 * k, re, im);
                    v[0] += re.x;
                    v[1] += im.x;
                    v[2] += re.y;
                    v[3] += im.y;
                }
            }
#pragma unroll
            for (int c = 0; c < 4; ++c) vs[4 * k + c] = v[c];
        }
        // the warp's 2 P sums by recursive halving: at offset o a lane keeps
        // the half of its values that its bit o selects (16 FP64 additions
        // instead of 80 for a shuffle tree per value)
        static_assert(2 * P == 16, "16 values, then one exchange between half warps");
#pragma unroll
        for (int lvl = 0; lvl < 4; ++lvl) {
            const int o = 1 << lvl, half = P >> lvl;
            const bool upper = (lane & o) != 0;
#pragma unroll
            for (int i = 0; i < half; ++i) {
                const double send = upper ? vs[i] : vs[i + half];
                const double keep = upper ? vs[i + half] : vs[i];
                vs[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
            }
        }
        vs[0] += __shfl_xor_sync(0xffffffffu, vs[0], 16);
        if (lane < 16) {  // lane bits 0..3 chose value bits 3..0
            const int i = ((lane & 1) << 3) | ((lane & 2) << 1) | ((lane & 4) >> 1) | (lane >> 3);
            red[i % 2][i / 2][warp] += vs[0];
        }
    }
    __syncthreads();
    if (threadIdx.x < P && p0 + (int)threadIdx.x < npts) {
        const int j = threadIdx.x;
        double a = 0.0, b = 0.0;
        for (int w = 0; w < kDirectThreads / 32; ++w) {
            a += red[0][j][w];
            b += red[1][j][w];
        }
        part[(size_t)blockIdx.y * npts + p0 + j] = make_double2(a, b);
    }
}

// The chunks' sums in order, times the outer factor: a warp per point.
__global__ void direct_finish_kernel(DirectGeom g, int form, int npts, const int* mx, const int* my,
                                     int chunks, const double2* part, const unsigned* bad, float2* out)
{
    chain_next();
    chain_wait();
    const int i = (int)(((size_t)blockIdx.x * blockDim.x + threadIdx.x) / 32);
    const int lane = threadIdx.x % 32;
    if (i >= npts) return;  // warp-uniform
    double a = 0.0, b = 0.0;
    for (int k = lane; k < chunks; k += 32) {
        const double2 v = part[(size_t)k * npts + i];
        a += v.x;
        b += v.y;
    }
    for (int o = 16; o > 0; o >>= 1) {
        a += __shfl_xor_sync(0xffffffffu, a, o);
        b += __shfl_xor_sync(0xffffffffu, b, o);
    }
    if (lane != 0) return;
    if (*bad) a = b = __longlong_as_double(0x7ff8000000000000ll);
    // outer factor o = f * exp(i pi ph) / i = f (sin(pi ph) - i cos(pi ph))
    const double wgt = g.p1x * g.p1y;
    double f, ph;
    if (form == kEq2) {
        f = wgt * g.z0 / g.lambda;
        ph = 0.0;
    } else {
        f = wgt / (g.lambda * g.z0);
        ph = 2.0 * g.z0 / g.lambda;
        if (form == kEq7) {
            const double x2 = ((double)mx[i] - g.m2x / 2) * g.p2x;
            const double y2 = ((double)my[i] - g.m2y / 2) * g.p2y;
            ph += (x2 * x2 + y2 * y2) / (g.lambda * g.z0);
        }
    }
    ph -= 2.0 * rint(0.5 * ph);
    double sp, cp;
    sincospi(ph, &sp, &cp);
    const double ore = f * sp, oim = -f * cp;
    out[i] = make_float2((float)(ore * a - oim * b), (float)(ore * b + oim * a));
}

}  // namespace

asfd_status direct_sum(const asfd_params* p, const double* d1, const float2* u1, int form,
                       int npts, const int* mx, const int* my, float2* out, cudaStream_t st)
{
    if (!p || !d1 || !u1 || npts < 0)
        return fail(ASFD_ERR_ARG, "NULL argument or negative point count");
    if (npts > 0 && (!mx || !my || !out)) return fail(ASFD_ERR_ARG, "NULL point or output array");
    if (form != 2 && form != 5 && form != 7)
        return fail(ASFD_ERR_ARG, "form must be 2, 5 or 7 (the paper's Eq. 2, 5 or 7)");
    if (p->n1x < 2 || p->n1y < 2 || p->m2x < 2 || p->m2y < 2 || p->n1x % 2 || p->n1y % 2 ||
        p->m2x % 2 || p->m2y % 2 || p->n1x > 65536 || p->n1y > 65536)
        return fail(ASFD_ERR_ARG, "n1x, n1y, m2x, m2y must be even, >= 2 (n1 <= 65536)");
    const double pos[] = {p->p1x, p->p1y, p->p2x, p->p2y, p->lambda, p->z0};
    for (double x : pos)
        if (!(std::isfinite(x) && x > 0.0))
            return fail(ASFD_ERR_ARG, "pitches, wavelength and z0 must be finite and > 0");
    if (!(std::isfinite(p->incidence_sx) && std::isfinite(p->incidence_sy) &&
          p->incidence_sx * p->incidence_sx + p->incidence_sy * p->incidence_sy < 1.0))
        return fail(ASFD_ERR_ARG, "incidence direction cosines need sx^2 + sy^2 < 1");
    if (!(std::isfinite(p->offset_x) && std::isfinite(p->offset_y)))
        return fail(ASFD_ERR_ARG, "source offsets must be finite");
    if (npts == 0) return ASFD_OK;
    const double sz = std::sqrt(1.0 - p->incidence_sx * p->incidence_sx -
                                p->incidence_sy * p->incidence_sy);
    DirectGeom g{p->n1x, p->n1y, p->m2x, p->m2y, p->p1x, p->p1y, p->p2x, p->p2y,
                 p->lambda, p->z0, p->incidence_sx, p->incidence_sy, sz, p->offset_x,
                 p->offset_y, 1.0 / p->lambda};
    const size_t n = (size_t)p->n1x * p->n1y;
    // chunks of samples: enough blocks for every SM
    int dev = 0, sms = 0;
    ASFD_CUDA(cudaGetDevice(&dev));
    ASFD_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    const int eq = form == 5 && p->p2x != p->p2y ? (int)kEq5Uneven : form;
    const size_t groups = ((size_t)npts + kDirectPoints - 1) / kDirectPoints;
    const size_t most = (n + kDirectThreads - 1) / kDirectThreads;  // rows of a single chunk
    size_t chunks = ((size_t)kDirectBlocks * sms + groups - 1) / groups;
    chunks = std::min(chunks, (most + 3) / 4);
    const size_t rows = (most + chunks - 1) / chunks;
    chunks = (most + rows - 1) / rows;
    DirectTerms* s = nullptr;
    const size_t bytes = sizeof(DirectTerms) * n + sizeof(double2) * chunks * npts + sizeof(unsigned);
    cudaError_t e = cudaMallocAsync(reinterpret_cast<void**>(&s), bytes, st);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return fail(ASFD_ERR_NOMEM, std::string("per-sample terms: ") + cudaGetErrorString(e));
    }
    double2* part = reinterpret_cast<double2*>(s + n);
    unsigned* bad = reinterpret_cast<unsigned*>(part + chunks * npts);
    e = cudaMemsetAsync(bad, 0, sizeof(unsigned), st);
    if (e == cudaSuccess)
        e = launch_chained(direct_prep_kernel,
                           dim3((unsigned)((p->n1x + 255) / 256),
                                (unsigned)((p->n1y + kPrepRows - 1) / kPrepRows)),
                           256, 0, st, g, d1, eq, s, bad);
    const dim3 grid((unsigned)groups, (unsigned)chunks);
    const size_t chunk = rows * kDirectThreads;
    using T = const DirectTerms*;
    if (e == cudaSuccess) {
        switch (eq) {
#define ASFD_DS(F)                                                                                      \
    case F:                                                                                             \
        e = launch_chained(direct_sum_kernel<F>, grid, kDirectThreads, 0, st, g, T(s), u1, npts, mx, my, \
                           chunk, part);                                                                \
        break;
            ASFD_DS(kEq2) ASFD_DS(kEq5) ASFD_DS(kEq5Uneven) ASFD_DS(kEq7)
#undef ASFD_DS
            default: break;
        }
    }
    if (e == cudaSuccess)
        e = launch_chained(direct_finish_kernel, dim3((unsigned)(((size_t)npts + 7) / 8)), 256, 0, st, g, eq,
                           npts, mx, my, (int)chunks, (const double2*)part, (const unsigned*)bad, out);
    const cudaError_t ef = cudaFreeAsync(s, st);
    if (e != cudaSuccess) return cuda_fail(e, "direct_sum_kernel launch");
    if (ef != cudaSuccess) return cuda_fail(ef, "cudaFreeAsync");
    return ASFD_OK;
}

}  // namespace asfd
