// Mono-exponential T2 maps of a recovered image series (Sec. IV-A: the paper's T2 maps are
// obtained by fitting a mono-exponential model to every pixel of the reconstructed series).
//
//   |x_n(r)| ~ A(r) exp(-t_n / T2(r))   over foreground pixels |x_0(r)| > frac * max_r |x_0(r)|,
//
// log-linear least squares for the initial (A, 1/T2), then Gauss-Newton steps on the un-logged
// residual (2 x 2 normal equations per pixel, columns scaled to unit norm before Cramer's rule),
// 1/T2 kept >= 1e-4 per ms. One thread per pixel, all in FP32. The foreground decision
// is taken in FP32 with separately rounded products and sums (no contraction), so a host that
// repeats it in FP32 reaches the same mask bit for bit.
#include <cmath>

#include "common.cuh"
#include "kernels.h"

namespace recon {

namespace {

constexpr int kThreads = 256;
constexpr int kT2Threads = 128;  // small images spread over more SMs

RECON_DEV float magnitude_rn(float2 v) {
    return __fsqrt_rn(__fadd_rn(__fmul_rn(v.x, v.x), __fmul_rn(v.y, v.y)));
}

// max_r |x_0(r)| into *amax (non-negative floats order like their bit patterns: atomicMax on
// the bits is exact and independent of the order of arrival).
__global__ void __launch_bounds__(kThreads)
frame0_max_kernel(const float2* __restrict__ x, size_t npix, unsigned int* __restrict__ amax) {
    float m = 0.f;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < npix;
         i += (size_t)gridDim.x * blockDim.x)
        m = fmaxf(m, magnitude_rn(x[i]));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0) atomicMax(amax, __float_as_uint(m));
}

// One pixel a thread, its NT >= T samples and the echo times in registers, the loops over frames
// unrolled without branches (a frame beyond T adds exact zeros): the exponentials of a step are then
// independent instructions. (A loop over T with an array of the largest T and the times read from the
// parameters ran one exponential after the other: 20 % issue.) A Gauss-Newton step is a function of
// (A, R) alone: once a step returns values that it had before, the remaining steps go round the same
// cycle, and only the steps left over modulo its length are run. The values are bitwise those of
// running them all; most pixels stand after five steps of 20, a few per cent go round in the last
// bits. 256x256x16, 20 steps: 31.7 -> 19 us.
// More than 32 frames (kLong): the times come from the parameters (a constant operand of the unrolled
// code), the logarithms are formed twice, and four frames beyond T are left out at a time, so that the
// 64 samples leave registers for five CTAs an SM and 33 frames do not pay for 64. 256x256x33, 20 steps:
// 73 us a call by the loop over T, 77 with all 64 samples and times in registers (166 a thread), now 54; 5 steps
// 44, 68 and 47.
template <int NT>
__global__ void __launch_bounds__(kT2Threads, NT > 32 ? 5 : 0)
t2fit_kernel(const float2* __restrict__ x, int T, size_t npix, T2Times tm, float frac,
             const unsigned int* __restrict__ amax, int n_gn, float* __restrict__ t2,
             float* __restrict__ amp) {
    const size_t px = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (px >= npix) return;
    const float thr = __fmul_rn(frac, __uint_as_float(amax[0]));
    constexpr bool kLong = NT > 32;
    float y[NT], tt[NT];
#pragma unroll
    for (int n = 0; n < NT; ++n) {
        y[n] = n < T ? magnitude_rn(x[(size_t)n * npix + px]) : 0.f;
        if constexpr (kLong) {
            tt[n] = tm.t[n];  // 0 beyond T
            continue;
        }
        const float t = n < T ? tm.t[n] : 0.f;
        asm volatile("mov.f32 %0, %1;" : "=f"(tt[n]) : "f"(t));  // stays in a register
    }
    if (!(y[0] > thr)) {
        t2[px] = __int_as_float(0x7fc00000);  // NaN: not foreground
        if (amp) amp[px] = __int_as_float(0x7fc00000);
        return;
    }
    constexpr float kRmin = 1e-4f;  // 1 / T2 >= 1e-4 per ms (T2 <= 1e4 ms)
    // log-linear initial guess: log y = log A - R t
    float tbar = 0.f, lbar = 0.f, ly[NT];
#pragma unroll
    for (int n = 0; n < NT; ++n) {
        if (kLong && n % 4 == 0 && n >= T) break;
        ly[n] = n < T ? logf(fmaxf(y[n], 1e-30f)) : 0.f;
        tbar += tt[n];  // 0 beyond T
        lbar += ly[n];
    }
    tbar /= T;
    lbar /= T;
    float sxy = 0.f, sxx = 0.f;
#pragma unroll
    for (int n = 0; n < NT; ++n) {
        if (kLong && n % 4 == 0 && n >= T) break;
        const float dt = n < T ? tt[n] - tbar : 0.f;
        const float l = !kLong ? ly[n] : n < T ? logf(fmaxf(y[n], 1e-30f)) : 0.f;
        sxy = fmaf(dt, l - lbar, sxy);
        sxx = fmaf(dt, dt, sxx);
    }
    float R = fmaxf(-sxy / sxx, kRmin);
    float A = expf(lbar + R * tbar);
    // the two states before and one of 1, 2, 4, ... steps ago (cycles of one, two and any length)
    float A1 = __int_as_float(0x7fc00000), R1 = A1, Ac = A1, Rc = A1;
    int len = 1, power = 1;
    for (int it = 0; it < n_gn; ++it) {
        const float A0 = A, R0 = R;
        float a11 = 0.f, a12 = 0.f, a22 = 0.f, g1 = 0.f, g2 = 0.f;
#pragma unroll
        for (int n = 0; n < NT; ++n) {
            if (kLong && n % 4 == 0 && n >= T) break;
            const float e = n < T ? expf(-tt[n] * R) : 0.f;
            const float model = A * e;
            const float res = model - y[n];
            const float jr = -tt[n] * model;
            a11 = fmaf(e, e, a11);
            a12 = fmaf(e, jr, a12);
            a22 = fmaf(jr, jr, a22);
            g1 = fmaf(e, res, g1);
            g2 = fmaf(jr, res, g2);
        }
        // the 2 x 2 system with both columns scaled to unit norm: [1 c; c 1], det (1-c)(1+c)
        if (a11 > 0.f && a22 > 0.f) {
            const float s1 = rsqrtf(a11), s2 = rsqrtf(a22);
            const float c = a12 * s1 * s2;
            const float det = (1.f - c) * (1.f + c);
            if (det > 1e-12f) {
                const float h1 = g1 * s1, h2 = g2 * s2;
                const float id = 1.f / det;
                A -= s1 * (h1 - c * h2) * id;
                R = fmaxf(R - s2 * (h2 - c * h1) * id, kRmin);
            }
        }
        if (A == A0 && R == R0) break;
        int cycle = 0;
        if (A == A1 && R == R1) cycle = 2;
        else if (A == Ac && R == Rc) cycle = len;
        if (cycle) {
            n_gn = it + 1 + (n_gn - 1 - it) % cycle;
            A1 = Ac = __int_as_float(0x7fc00000);  // found: only the rest is run
            continue;
        }
        A1 = A0;
        R1 = R0;
        if (len == power) {
            Ac = A;
            Rc = R;
            power *= 2;
            len = 0;
        }
        ++len;
    }
    t2[px] = 1.0f / R;
    if (amp) amp[px] = A;
}

}  // namespace

cudaError_t launch_t2fit(const Dims& d, const float2* x, const T2Times& tm, float frac, int n_gn,
                         unsigned int* amax_scratch, float* t2, float* amp, cudaStream_t st) {
    if (d.T < 2 || d.T > kT2MaxT) return cudaErrorInvalidValue;
    const size_t npix = d.pixels();
    cudaError_t e = cudaMemsetAsync(amax_scratch, 0, sizeof(unsigned int), st);
    if (e != cudaSuccess) return e;
    const int g0 = (int)((npix + kThreads - 1) / kThreads < 1024 ? (npix + kThreads - 1) / kThreads : 1024);
    frame0_max_kernel<<<g0, kThreads, 0, st>>>(x, npix, amax_scratch);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const int g1 = (int)((npix + kT2Threads - 1) / kT2Threads);
#define CASE(NT)                                                                                  \
    if (d.T <= NT) {                                                                              \
        t2fit_kernel<NT><<<g1, kT2Threads, 0, st>>>(x, d.T, npix, tm, frac, amax_scratch, n_gn,   \
                                                    t2, amp);                                     \
        return cudaGetLastError();                                                                \
    }
    CASE(4) CASE(8) CASE(12) CASE(16) CASE(20) CASE(24) CASE(32) CASE(64)
#undef CASE
    return cudaErrorInvalidValue;
}

}  // namespace recon
