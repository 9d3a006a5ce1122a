// CG operator tail, CG vector updates and the warm-start residual carry (Sec. III-A,
// Eq. grad-ls; Algorithm 1, step 2).
//
// The sum-of-squares weight acts per pixel r as a banded frame operator built from the M x M
// Hermitian matrix S(r) (the precomputed G of Eq. grad-ls, the sum of k shifted copies of one
// block product):
//     (W x)_n(r) = sum_{a : 0 <= n-M+1+a < k} sum_b S_ab(r) x_{n+a-b}(r),
// which is sum_j E_j^T S(r) E_j x(r) with (E_j x)(r)[m] = x_{j+M-1-m}(r). S is stored as its
// upper triangle, pair (a <= b) at index a(2M-a+1)/2 + (b-a), layout [pair][P][Q] complex64.
#include <map>
#include <mutex>
#include <tuple>

#include "common.cuh"
#include "kernels.h"
#include "regfft.cuh"
#include "stockham.cuh"

namespace recon {

namespace {

constexpr int kThreads = 256;
constexpr int kMaxM = 6;
// Dynamic shared memory that needs no opt-in next to a kernel's static arrays (48 KB for both).
constexpr size_t kDynSmemFree = 40 * 1024;
constexpr int kMaxParts = 4096;  // partial-sum slots (largest grid of a reducing kernel)
constexpr int kUpdVec = 2;       // float4 per thread per iteration in the update pass
constexpr int kUpdThreads = 512;
constexpr int kUpdPerSM = 2;     // update CTAs per SM (few partials for the next pass to add)

// Load S(r) (full M x M from the stored upper triangle) into registers.
template <int M>
RECON_DEV void load_S(const float2* __restrict__ S, size_t npix, size_t px, float2 (&s)[M][M]) {
#pragma unroll
    for (int a = 0; a < M; ++a)
#pragma unroll
        for (int b = a; b < M; ++b) {
            const float2 v = S[(size_t)(a * (2 * M - a + 1) / 2 + (b - a)) * npix + px];
            s[a][b] = v;
            s[b][a] = cconj(v);
        }
}

// Diagonal sums of the per-pixel block: c[M - 1 + d] = sum_{a - b = d} s[a][b], d = -(M-1) ..
// M-1. A frame n whose M windows n - M + 1 + a all exist (every frame of the circular lifting)
// has (W x)_n = sum_d c[M - 1 + d] x_{n+d}: 2M - 1 products instead of M^2. s is Hermitian, so
// c[M - 1 - d] = conj(c[M - 1 + d]).
template <int M>
RECON_DEV void s_diagonals(const float2 (&s)[M][M], float2 (&c)[2 * M - 1]) {
#pragma unroll
    for (int d = 0; d < M; ++d) {
        float2 v = make_float2(0.f, 0.f);
#pragma unroll
        for (int a = d; a < M; ++a) v = cadd(v, s[a][a - d]);
        c[M - 1 + d] = v;
        if (d > 0) c[M - 1 - d] = cconj(v);
    }
}

// Row transforms of pass C: kIn elements i + m kLanes of a row in u[m] on entry, element out_at(i, m) of
// the result in u[m] on return; rows of 128 and 256 elements by the two-stage transforms of regfft.cuh
// (16 elements a thread, one exchange), the others by the Stockham passes.
template <int N>
struct RowFft : RegFft<N> {
    static constexpr int kIn = 8;
    static constexpr bool kByWarp = false;
    RECON_DEV static void fill(float2* tw, const float2* __restrict__ tw_g) {
        for (int i = threadIdx.x; i < N; i += blockDim.x) tw[i] = tw_g[i];
    }
    RECON_DEV static void inverse(float2 (&u)[RegFft<N>::kOut], float2* sx, const float2* tw, int i) {
        RegFft<N>::template run<true, false>(u, sx, 1, tw, i);
    }
};
template <int N>
struct RowFft16 {
    static constexpr int kLanes = N / 16, kIn = 16, kOut = 16;
    static constexpr bool kByWarp = true;  // warps without a frame leave the transform out
    RECON_DEV static void sync() { __syncwarp(); }
};
template <>
struct RowFft<256> : RowFft16<256> {
    static constexpr int kBuf = 16 * 17;
    RECON_DEV static int out_at(int i, int m) { return i + 16 * m; }
    RECON_DEV static int at(int e) { return e + (e >> 4); }
    RECON_DEV static void fill(float2* tw, const float2* __restrict__ tw_g) { fill_tw256(tw, tw_g); }
    RECON_DEV static void inverse(float2 (&u)[16], float2* sx, const float2* tw, int i) {
        row_dft256<true>(u, sx, tw, i);
    }
};
template <>
struct RowFft<128> : RowFft16<128> {
    static constexpr int kBuf = kX128;
    RECON_DEV static int out_at(int i, int m) { return 2 * i + (m & 1) + 16 * (m >> 1); }
    RECON_DEV static int at(int e) { return e + (e >> 3); }
    RECON_DEV static void fill(float2* tw, const float2* __restrict__ tw_g) { fill_tw128(tw, tw_g); }
    RECON_DEV static void inverse(float2 (&u)[16], float2* sx, const float2* tw, int i) {
        float2 a[8], b[8];
        row_dft128<true>(u, a, b, sx, tw, i);
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            u[2 * k] = a[k];
            u[2 * k + 1] = b[k];
        }
    }
};

// The W phase of pass C for frames [n0, n1) of one image row, by the whole CTA: res[n - n0][at(c)]
// holds the transformed rows; q = res + lam W p goes to t, and Re (conj p) q of every element takes the
// place of res.
// A thread takes a column and a run of FC frames, whose p values and the M - 1 on either side it reads
// straight from global memory into registers (each once per run; no copy of the p rows in shared
// memory). kDiag: the diagonal form where all M windows of a frame exist (for 3 <= M <= 5, where it saves
// products and the block and its sums fit the registers; the circular lifting always).
// kAhead: the loads of a thread's first task (WLoads) were issued before the transform of the rows; for rows
// of 128 and more elements up to three taps, more do not fit the registers next to the transform's elements
// (256x256x16, M = 4: 220 bytes of spills at 80 registers).
// Runs of eight frames for rows of 128 and 256 elements, and for long rows with more than four taps, whose
// M - 1 frames on either side and M (M + 1) / 2 weights a run are the most of its loads: runs of two took
// 36.1 us a CG step at 256x256x16, M = 5, eight take 27.0 (M = 6: 39.5 and 29.9; 512x512x16: 176 and 142).
// Rows of up to 64 elements are bound by latency: more, shorter tasks (128x16x126, M = 5: 15 steps 353 us with
// runs of two frames, 440 with four).
template <class F, int M>
constexpr int kWRun = F::kIn > 8 ? 8 : M <= 4 ? 4 : F::kLanes <= 8 ? 2 : 8;
template <class F, int M>
constexpr bool kWAhead = M <= 3 || (F::kIn <= 8 && F::kLanes <= 8);
template <int M, int FC>
struct WLoads {
    float2 pw[FC + 2 * (M - 1)];    // p_{f0 - (M - 1) + i}
    float2 s[M * (M + 1) / 2];      // upper triangle of S(r)
};
template <int N, int M, int FC, bool CIRC>
RECON_DEV void w_load(WLoads<M, FC>& v, const float2* __restrict__ prow, const float2* __restrict__ Srow,
                      int e, int T, int n0, int n1, size_t npix) {
    const int c = e % N, f0 = n0 + (e / N) * FC, f1 = min(n1, f0 + FC);
#pragma unroll
    for (int i = 0; i < FC + 2 * (M - 1); ++i) {
        const int f = f0 - (M - 1) + i;
        v.pw[i] = make_float2(0.f, 0.f);
        if (f0 < n1 && f < f1 + M - 1 && (CIRC || (f >= 0 && f < T)))
            v.pw[i] = prow[(size_t)(CIRC ? wrap_frame(f, T) : f) * npix + c];
    }
#pragma unroll
    for (int i = 0; i < M * (M + 1) / 2; ++i) v.s[i] = Srow[(size_t)i * npix + c];
}

template <class F, int N, int M, int FC, bool CIRC, bool kDiag, bool kAhead>
RECON_DEV void w_phase(WLoads<M, FC>& v, float2* __restrict__ trow, const float2* __restrict__ prow,
                       const float2* __restrict__ Srow, float2* res, float lam, int T, int n0, int n1,
                       size_t npix) {
    const int k = CIRC ? T : T - M + 1;
    const int nrun = (n1 - n0 + FC - 1) / FC;
    for (int e = threadIdx.x; e < N * nrun; e += blockDim.x) {
        if (!kAhead || e != (int)threadIdx.x) w_load<N, M, FC, CIRC>(v, prow, Srow, e, T, n0, n1, npix);
        const int c = e % N, f0 = n0 + (e / N) * FC, f1 = min(n1, f0 + FC);
        float2 s[M][M];
#pragma unroll
        for (int a = 0; a < M; ++a)
#pragma unroll
            for (int b = a; b < M; ++b) {
                s[a][b] = v.s[a * (2 * M - a + 1) / 2 + (b - a)];
                s[b][a] = cconj(s[a][b]);
            }
        float2 cs[2 * M - 1];
        if constexpr (kDiag) s_diagonals<M>(s, cs);
#pragma unroll
        for (int i = 0; i < FC; ++i) {
            const int n = f0 + i;
            if (n >= f1) break;
            float2 w = make_float2(0.f, 0.f);
            if (kDiag && (CIRC || (M >= 3 && M <= 5 && n >= M - 1 && n < k))) {
#pragma unroll
                for (int d = 0; d < 2 * M - 1; ++d) w = cfma(cs[d], v.pw[i + d], w);
            } else {
#pragma unroll
                for (int a = 0; a < M; ++a) {
                    const int j = n - M + 1 + a;
                    if (j < 0 || j >= k) continue;
#pragma unroll
                    for (int b = 0; b < M; ++b) w = cfma(s[a][b], v.pw[i + M - 1 + a - b], w);
                }
            }
            float2* rp = res + (size_t)(n - n0) * F::kBuf + F::at(c);
            float2 q = *rp;
            q.x = fmaf(lam, w.x, q.x);
            q.y = fmaf(lam, w.y, q.y);
            trow[(size_t)n * npix + c] = q;
            const float2 pv = v.pw[i + M - 1];
            rp->x = fmaf(pv.x, q.x, pv.y * q.y);
        }
    }
}

// The terms that w_phase left, added per column over the frames in order (Kahan), and over the columns
// by FP32 warp trees: a warp's sum in its lane 0, FP64, zero elsewhere. Columns c and c + kThreads share
// an accumulator, so that the sum of a run is that of a CTA of kThreads threads, one column each, whatever
// the CTA's threads (CG amplifies the last bits of Re <p, q> on the smallest series).
template <class F, int N>
RECON_DEV double w_terms(const float2* res, int T) {
    const int nc = N < kThreads ? N : kThreads;
    double tot = 0.0;
    for (int c0 = 0; c0 < nc; c0 += blockDim.x) {
        float acc = 0.f, comp = 0.f;
        if (c0 + (int)threadIdx.x < nc) {
            for (int c = c0 + threadIdx.x; c < N; c += kThreads)
                for (int n = 0; n < T; ++n) {
                    const float term = res[(size_t)n * F::kBuf + F::at(c)].x - comp;
                    const float sum = acc + term;
                    comp = (sum - acc) - term;
                    acc = sum;
                }
        }
        tot += (double)warp_sum(acc);
    }
    return tot;
}

// Sum over the CTA's warps of a value held by every lane 0 (thread 0 gets it).
RECON_DEV double warps_sum_t0(double v, double* red) {
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    double t = 0.0;
    if (threadIdx.x < 32) {
        t = threadIdx.x < blockDim.x / 32 ? red[threadIdx.x] : 0.0;
        t = warp_sum(t);
    }
    return t;
}

// Launch shape of the row passes that hold every frame of an image row: the frames in `passes` equal
// parts of at most inv_threads / (N / 8) sequences, whole warps; `bufs` exchange buffers.
template <int N>
__host__ __device__ constexpr int inv_threads() { return N == 192 ? 384 : 512; }
struct InvShape {
    int passes, per, threads, bufs;
};
template <int N>
InvShape inv_shape(int T) {
    constexpr int L = RegFft<N>::kLanes;
    InvShape v;
    v.passes = (T * L + inv_threads<N>() - 1) / inv_threads<N>();
    v.per = (T + v.passes - 1) / v.passes;
    v.threads = (v.per * L + 31) / 32 * 32;
    if (v.threads < 64) v.threads = 64;
    v.bufs = (v.passes - 1) * v.per + (v.threads + L - 1) / L;
    return v;
}

// Pass C of a CG step. A CTA takes a run of `per` frames of an image row r1 (W reads the neighbouring
// frames' p from global memory, so the runs are independent), kLanes threads per frame: it
// inverse-transforms the k-space rows of t (giving A^H A p; the 1/(PQ) scale was applied with the mask;
// elements in registers, exchange buffers that then hold the transformed rows), adds lam W p, writes q
// over t and emits a partial of Re <p, q>. Rows of up to 32 elements keep all their frames in one CTA, up
// to 256 frames of 16-point and 128 of 32-point rows, and with it the order of that sum (see w_terms). The pass is bound by latency for image series, by HBM
// for volumes. 64x64x21 7.8 -> 4.4 us per launch, 192x192x24 17.4 -> 9.6, 512x512x16 66.6 -> 32.3,
// against one CTA per row with passes over shared memory and three copies of the row's frames there.
// Rows of 128 and 256 elements took such copies of p (and of t and S) too, with asynchronous staging
// for volumes: without them and with W in runs of eight frames a volume of 128x128x64x12 (2 x 15 steps)
// takes 10.5 instead of 11.2 ms, four 256x256x16 solves at once 16.6 instead of 17.9, a single one the
// same 19.2, 15 steps at 512x128x12 508 instead of 548 us. Registers decide: 80 let two CTAs of 24
// 256-point frames share an SM (at 128: 671 us for 15 steps at 256x256x24 instead of 633).
// Most threads of a CTA. 192-point rows with up to four taps: 16 frames, so that series of 11 to 16 frames
// need no second run (512x192x11, M = 4: 41.2 us a step with two runs, 37.8 with one); 512-point rows with
// more: eight frames for the same reason (256x512x5, M = 5: 33.1 us with two runs, 30.4 with one).
template <int N, int M>
__host__ __device__ constexpr int run_threads() {
    return N <= 32 || (N == 512 && M > 4) ? 512 : N == 256 || (N == 192 && M <= 4) ? 384 : 256;
}
// CTAs an SM that the registers are held to. More than four taps with 16 elements a thread take 117 to 128
// registers, one CTA of 256-point rows (256x256x24, M = 5: 41.5 us a step, 43.9 at 80 registers with spills).
template <int N, int M>
__host__ __device__ constexpr int run_blocks() {
    if (N <= 32) return 1;
    if (M > 4) return N == 192 ? 2 : 1;
    return N == 256 || N == 192 || (N == 128 && M == 4) ? 2 : 3;
}
// Units wanted (CTAs of the shortest runs that fit the chip at once), and frames of the shortest run: eight
// for 256-point rows and for long rows with more than four taps, as many as a thread of W takes at once; else four.
// (128x256x5 and x8, M = 3: 14.9 and 14.8 us a step with runs of four frames, 14.0 and 14.3 with one run. With
// fewer than 128 image rows four: 64x256x24 16.0 us with 256 units, 17.2 with 192.)
template <int N>
constexpr int kRunUnits = N == 256 ? 456 : N == 128 ? 304 : 608;
struct RunShape {
    int nrun, per, threads, bufs;
};
template <class F, int N, int M>
RunShape run_shape(int T, int rows) {
    constexpr int L = F::kLanes;
    // Frames of a CTA in whole sequences: 24 threads a frame (192-point rows) do not divide the CTA's
    // threads, and a share of 256 / 24 frames rounded up would ask for more than there are. Series of more
    // than 16 frames of 192-point rows in runs of ten at most (256x192x24: 32.0 us a step, 34.0 with 12).
    constexpr int most_frames = run_threads<N, M>() / L;
    // W's tasks come in rounds of the CTA's threads: half a row more or less, so that no round is nearly
    // empty (21 frames of 256-point rows: 768 tasks, two rounds of 384 threads or three of 352)
    constexpr int grain = F::kIn > 8 ? N / 2 : 32;
    static_assert((most_frames * L + grain - 1) / grain * grain <= run_threads<N, M>() &&
                      64 <= run_threads<N, M>() && (F::kIn <= 8 || N <= run_threads<N, M>()),
                  "a run's threads exceed the kernel's launch bounds");
    RunShape v;
    const int most = N == 192 && T > 16 && most_frames > 10 ? 10 : most_frames;
    int n = (T + most - 1) / most;
    if (N > 32) {  // more, shorter runs until the units fill the chip
        // (rounded down: a few units more than fit at once would take a second round of their own)
        const int shortest = (N == 256 && rows >= 128) || (N > 64 && M > 4) ? 8 : 4;
        const int fill = (N == 256 && rows < 128 ? 304 : kRunUnits<N>) / rows, limit = (T + shortest - 1) / shortest;
        if (n < fill) n = fill < limit ? fill : (n > limit ? n : limit);
    }
    v.per = (T + n - 1) / n;
    v.nrun = (T + v.per - 1) / v.per;
    v.threads = (v.per * L + 31) / 32 * 32;
    if (v.threads < 64) v.threads = 64;
    v.bufs = (v.threads + L - 1) / L;
    // Rows of 128 and 256 elements: at least a thread per column for W (128x128x12, M = 3: 340 us for 15
    // steps with 64 threads, 326 with 128); warps without a frame have no part in the transform.
    if (F::kIn > 8 && v.threads < N) v.threads = N;
    v.threads = (v.threads + grain - 1) / grain * grain;
    return v;
}

template <class F, int N, int M, bool CIRC>
__global__ void __launch_bounds__((run_threads<N, M>()), (run_blocks<N, M>()))
row_inv_w_kernel(float2* t, const float2* __restrict__ p, const float2* __restrict__ S,
                 float lam, int T, int P, int nrun, int per, double* __restrict__ pq_parts,
                 const float2* __restrict__ tw_g) {
    extern __shared__ float2 sm[];
    __shared__ double red[16];
    float2* tw = sm;
    float2* res = sm + N;
    const size_t npix = (size_t)P * N;
    F::fill(tw, tw_g);
    const int fl = threadIdx.x / F::kLanes, i = threadIdx.x % F::kLanes;
    float2* sx = res + fl * F::kBuf;
    pdl_wait();
    double tot = 0.0;
    __syncthreads();  // tw
    const int nunit = P * nrun;
    for (int un = blockIdx.x; un < nunit; un += gridDim.x) {
        const int r1 = un / nrun, n0 = (un % nrun) * per, n1 = min(T, n0 + per);
        float2* trow = t + (size_t)r1 * N;
        const bool ok = n0 + fl < n1;
        float2 u[F::kOut];
#pragma unroll
        for (int m = 0; m < F::kIn; ++m)
            u[m] = ok ? trow[(size_t)(n0 + fl) * npix + i + m * F::kLanes] : make_float2(0.f, 0.f);
        constexpr int FC = kWRun<F, M>;
        WLoads<M, FC> wl;
        if constexpr (kWAhead<F, M>)
            w_load<N, M, FC, CIRC>(wl, p + (size_t)r1 * N, S + (size_t)r1 * N, threadIdx.x, T, n0, n1, npix);
        if (!F::kByWarp || n0 + (int)(threadIdx.x & ~31u) / F::kLanes < n1) {
            F::inverse(u, sx, tw, i);
            F::sync();  // the last exchange is read
#pragma unroll
            for (int m = 0; m < F::kOut; ++m) {
                const int e = F::out_at(i, m);
                if (e >= 0) sx[F::at(e)] = u[m];
            }
        }
        __syncthreads();
        w_phase<F, N, M, FC, CIRC, true, kWAhead<F, M>>(wl, trow, p + (size_t)r1 * N, S + (size_t)r1 * N, res,
                                                         lam, T, n0, n1, npix);
        __syncthreads();  // the terms
        if (un + (int)gridDim.x >= nunit) pdl_trigger();
        tot += w_terms<F, N>(res, n1 - n0);
        __syncthreads();  // the terms are read
    }
    tot = warps_sum_t0(tot, red);
    if (threadIdx.x == 0) pq_parts[blockIdx.x] = tot;
}

// Pass C of a CG step with coils (ADJ = false), or the coil combination of the adjoint
// (ADJ = true). One CTA per image row r1, N / 8 threads per frame: for each coil c they
// inverse-transform the row t[c][n][r1] and accumulate conj(C_c) * (...) in registers, the next coil's
// row in flight meanwhile (Eq. measurement-ij: A^H = sum_c conj(C_c) F^H mask). ADJ: the sum is
// x[n][r1]. Otherwise lam W p is added as in row_inv_w_kernel, q goes over coil 0's plane of t (rows r1,
// read by this CTA only) and the row's partial Re <p, q> to pq_parts. 12 coils at 128x128x12: 42.3 ->
// 12.5 us per launch, against a block barrier after every pass of every coil.
template <int N, int M, bool ADJ>
__global__ void __launch_bounds__(inv_threads<N>())
coil_row_inv_kernel(float2* t, const float2* __restrict__ p, const float2* __restrict__ coils,
                    const float2* __restrict__ S, float lam, int T, int P, int nc, int passes, int per,
                    double* __restrict__ pq_parts, float2* __restrict__ x_out,
                    const float2* __restrict__ tw_g) {
    using F = RegFft<N>;
    extern __shared__ float2 sm[];
    __shared__ double red[16];
    float2* tw = sm;
    float2* res = sm + N;
    const int r1 = blockIdx.x;
    const size_t npix = (size_t)P * N;
    const size_t series = (size_t)T * npix;
    for (int i = threadIdx.x; i < N; i += blockDim.x) tw[i] = tw_g[i];
    const int fl = threadIdx.x / F::kLanes, i = threadIdx.x % F::kLanes;
    pdl_wait();
    __syncthreads();  // tw
    float2* trow = t + (size_t)r1 * N;
    const float2* crow = coils + (size_t)r1 * N;
    for (int ps = 0; ps < passes; ++ps) {
        const int n = ps * per + fl;
        const bool ok = fl < per && n < T;
        float2* sx = res + (size_t)n * F::kBuf;
        float2 acc[F::kOut], nx[8];
#pragma unroll
        for (int m = 0; m < F::kOut; ++m) acc[m] = make_float2(0.f, 0.f);
#pragma unroll
        for (int m = 0; m < 8; ++m)
            nx[m] = ok ? trow[(size_t)n * npix + i + m * F::kLanes] : make_float2(0.f, 0.f);
        for (int c = 0; c < nc; ++c) {
            float2 u[F::kOut], cv[F::kOut];
#pragma unroll
            for (int m = 0; m < 8; ++m) u[m] = nx[m];
            if (c + 1 < nc && ok) {
#pragma unroll
                for (int m = 0; m < 8; ++m)
                    nx[m] = trow[(size_t)(c + 1) * series + (size_t)n * npix + i + m * F::kLanes];
            }
#pragma unroll
            for (int m = 0; m < F::kOut; ++m) {
                const int e = F::out_at(i, m);
                cv[m] = e >= 0 ? crow[(size_t)c * npix + e] : make_float2(0.f, 0.f);
            }
            F::sync();  // the previous coil's last exchange is read
            F::template run<true, false>(u, sx, 1, tw, i);
#pragma unroll
            for (int m = 0; m < F::kOut; ++m) acc[m] = cfmacj(cv[m], u[m], acc[m]);
        }
        if constexpr (ADJ) {
            if (ok) {
#pragma unroll
                for (int m = 0; m < F::kOut; ++m) {
                    const int e = F::out_at(i, m);
                    if (e >= 0) x_out[(size_t)n * npix + (size_t)r1 * N + e] = acc[m];
                }
            }
        } else {
            F::sync();
#pragma unroll
            for (int m = 0; m < F::kOut; ++m) {
                const int e = F::out_at(i, m);
                if (e >= 0) sx[F::at(e)] = acc[m];
            }
        }
        // spare threads of a pass share the next pass's first buffers
        if (ps + 1 < passes) __syncthreads();
    }
    if constexpr (ADJ) {
        pdl_trigger();
        return;
    } else {
        __syncthreads();
        constexpr int FC = M > 4 ? 2 : 4;
        WLoads<M, FC> wl;
        w_load<N, M, FC, false>(wl, p + (size_t)r1 * N, S + (size_t)r1 * N, threadIdx.x, T, 0, T, npix);
        w_phase<F, N, M, FC, false, false, true>(wl, trow, p + (size_t)r1 * N, S + (size_t)r1 * N, res, lam, T, 0, T, npix);
        __syncthreads();  // the terms
        pdl_trigger();
        const double tot = warps_sum_t0(w_terms<F, N>(res, T), red);
        if (threadIdx.x == 0) pq_parts[blockIdx.x] = tot;
    }
}

// Pass D: alpha = |r|^2 / Re <p, q> (Re <p, q> summed here from pass C's partials), stored for the next
// pass A; r -= alpha q; per-CTA partials of |r_new|^2 for the next pass A; x += alpha p with kX (else
// the next pass A does it). Bound by memory (L2 or HBM), 256x256x16 7.5 us with x; the order of the sum
// is the same with and without x.
template <bool kX>
__global__ void __launch_bounds__(kUpdThreads, kUpdPerSM)
cg_update_kernel(float4* __restrict__ x, float4* __restrict__ r, const float4* __restrict__ p,
                 const float4* __restrict__ q, size_t n4, const double* __restrict__ rr_in,
                 const double* __restrict__ pq_parts, int n_pq, double* __restrict__ rr_parts,
                 double* __restrict__ alpha_out) {
    constexpr int V = kX ? kUpdVec : 2 * kUpdVec;
    __shared__ double red[kUpdThreads / 32];
    __shared__ double s_pq;
    __shared__ float alpha_s;
    pdl_wait();
    const size_t stride = (size_t)gridDim.x * blockDim.x;
    size_t i0 = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    float4 xv[V], rv[V], pv[V], qv[V];
    auto load = [&](size_t at) {
#pragma unroll
        for (int u = 0; u < V; ++u) {
            const size_t i = at + (size_t)u * stride;
            if (i >= n4) continue;
            rv[u] = r[i];
            qv[u] = q[i];
            if constexpr (kX) {
                xv[u] = x[i];
                pv[u] = p[i];
            }
        }
    };
    load(i0);  // the first loads go out before alpha is known (they do not depend on it)
    const double pq = sum_partials(pq_parts, n_pq, &s_pq);
    if (threadIdx.x == 0) {
        alpha_s = (float)(rr_in[0] * rcp_nr(pq));
        if (blockIdx.x == 0) alpha_out[0] = (double)alpha_s;
    }
    __syncthreads();
    const float alpha = alpha_s;
    float acc = 0.f, comp = 0.f;
    for (; i0 < n4; i0 += stride * V) {
#pragma unroll
        for (int u = 0; u < V; ++u) {
            const size_t i = i0 + (size_t)u * stride;
            if (i >= n4) continue;
            if constexpr (kX) {
                xv[u].x = fmaf(alpha, pv[u].x, xv[u].x);
                xv[u].y = fmaf(alpha, pv[u].y, xv[u].y);
                xv[u].z = fmaf(alpha, pv[u].z, xv[u].z);
                xv[u].w = fmaf(alpha, pv[u].w, xv[u].w);
                x[i] = xv[u];
            }
            rv[u].x = fmaf(-alpha, qv[u].x, rv[u].x);
            rv[u].y = fmaf(-alpha, qv[u].y, rv[u].y);
            rv[u].z = fmaf(-alpha, qv[u].z, rv[u].z);
            rv[u].w = fmaf(-alpha, qv[u].w, rv[u].w);
            r[i] = rv[u];
            const float4 w = rv[u];
            const float term = fmaf(w.x, w.x, fmaf(w.y, w.y, fmaf(w.z, w.z, w.w * w.w))) - comp;
            const float sum = acc + term;
            comp = (sum - acc) - term;
            acc = sum;
        }
        load(i0 + stride * V);
    }
    pdl_trigger();
    const double tot = block_sum_f_t0(acc, red);
    if (threadIdx.x == 0) rr_parts[blockIdx.x] = tot;
}

__global__ void sum_partials_kernel(const double* __restrict__ parts, int n, double* __restrict__ out) {
    const double v = warp0_sum_array(parts, n);
    if (threadIdx.x == 0) out[0] = v;
}

// Residual carry between IRLS iterations: r = (first ? r0 : r) + lam W_{dS} x with
// dS = S_old - S_new (or -S_new when first); partial |r|^2.
// r0 = A^H b - A^H A x0 = x0 - A^H A x0 for x0 = A^H b: zero for one coil and 0/1 masks (A A^H
// is then a projection), x0 - aha_x when A^H A x0 is supplied (coils).
// A warp takes 32 pixels and a run of up to FC frames, whose x values and the M - 1 on either side are
// held in registers (one read of each instead of M^2; the order of the window sum does not depend on
// the runs). The runs of a pixel group are warps of one CTA; the squares of a pixel meet in shared
// memory and are added over the frames in order, so that |r|^2 does not depend on the runs either:
// CG amplifies its last bits on the smallest series. The kernel runs once per IRLS iteration and is
// bound by latency for small series, by memory for large ones: FC trades the warps in flight against
// the re-reading of S and of the frames at a run's ends (resid_run below). 64x64x21, M = 2: 14.0 ->
// 7.7 us; 256x256x16, M = 3: 15.4 -> 12.8; 128x128x64x12, M = 2: 82 -> 68 (one thread a
// pixel with all frames before).
constexpr int kResWarps = 8;  // most warps of a CTA
template <int M, int FC>
__global__ void __launch_bounds__(32 * kResWarps)
resid_carry_kernel(float2* __restrict__ r, const float2* __restrict__ x,
                   const float2* __restrict__ aha_x, const float2* __restrict__ S_old,
                   const float2* __restrict__ S_new, float lam, int first, int T, int circ,
                   size_t npix, int nrun, int run, int nwr, double* __restrict__ parts,
                   unsigned int* counter, double* __restrict__ rr_out) {
    extern __shared__ float terms[];  // [pixel group of the CTA][T][32] where a pixel has several runs
    __shared__ double red[kResWarps];
    pdl_wait();
    const int k = circ ? T : T - M + 1;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int ngrp = (blockDim.x >> 5) / nwr, grp = warp / nwr;  // pixel groups per CTA, nwr warps each
    float* tg = terms + (size_t)grp * T * 32 + lane;
    const size_t npg = npix / 32;  // P and Q are multiples of 16
    double tot = 0.0;
    for (size_t g0 = (size_t)blockIdx.x * ngrp; g0 < npg; g0 += (size_t)gridDim.x * ngrp) {
        const size_t px = (g0 + grp) * 32 + lane;
        const bool live = g0 + grp < npg;
        float acc = 0.f, comp = 0.f;
        for (int rn = warp % nwr; live && rn < nrun; rn += nwr) {
            const int f0 = rn * run, f1 = min(T, f0 + run);
            float2 xw[FC + 2 * (M - 1)], rv[FC];  // x_{f0 - (M - 1) + i}, r_{f0 + i}
#pragma unroll
            for (int i = 0; i < FC + 2 * (M - 1); ++i) {
                const int f = f0 - (M - 1) + i;
                xw[i] = make_float2(0.f, 0.f);
                if (f < f1 + M - 1 && (circ || (f >= 0 && f < T)))
                    xw[i] = x[(size_t)wrap_frame(f, T) * npix + px];
            }
#pragma unroll
            for (int i = 0; i < FC; ++i) {
                rv[i] = make_float2(0.f, 0.f);
                if (f0 + i >= f1) continue;
                const size_t g = (size_t)(f0 + i) * npix + px;
                if (!first) {
                    rv[i] = r[g];
                } else if (aha_x) {  // x0 - A^H A x0 (coils: A A^H is no projection)
                    const float2 av = aha_x[g];
                    rv[i] = make_float2(xw[i + M - 1].x - av.x, xw[i + M - 1].y - av.y);
                }
            }
            float2 s[M][M];
            load_S<M>(S_new, npix, px, s);
            if (first) {
#pragma unroll
                for (int a = 0; a < M; ++a)
#pragma unroll
                    for (int b = 0; b < M; ++b) s[a][b] = make_float2(-s[a][b].x, -s[a][b].y);
            } else {
                float2 so[M][M];
                load_S<M>(S_old, npix, px, so);
#pragma unroll
                for (int a = 0; a < M; ++a)
#pragma unroll
                    for (int b = 0; b < M; ++b) s[a][b] = csub(so[a][b], s[a][b]);
            }
#pragma unroll
            for (int i = 0; i < FC; ++i) {
                const int n = f0 + i;
                if (n >= f1) break;
                float2 w = make_float2(0.f, 0.f);
#pragma unroll
                for (int a = 0; a < M; ++a) {
                    const int j = n - M + 1 + a;
                    if (!circ && (j < 0 || j >= k)) continue;  // circ: every window
#pragma unroll
                    for (int b = 0; b < M; ++b) w = cfma(s[a][b], xw[i + M - 1 + a - b], w);
                }
                rv[i].x = fmaf(lam, w.x, rv[i].x);
                rv[i].y = fmaf(lam, w.y, rv[i].y);
                r[(size_t)n * npix + px] = rv[i];
                const float sq = fmaf(rv[i].x, rv[i].x, rv[i].y * rv[i].y);
                if (nrun > 1) {
                    tg[n * 32] = sq;
                } else {
                    const float term = sq - comp;
                    const float sum = acc + term;
                    comp = (sum - acc) - term;
                    acc = sum;
                }
            }
        }
        if (nrun > 1) {
            __syncthreads();
            for (int n = 0; warp % nwr == 0 && live && n < T; ++n) {
                const float term = tg[n * 32] - comp;
                const float sum = acc + term;
                comp = (sum - acc) - term;
                acc = sum;
            }
            __syncthreads();  // the terms are read
        }
        tot += (double)warp_sum(acc);  // zero in the warps of later runs
    }
    pdl_trigger();
    if (lane == 0) red[warp] = tot;
    __syncthreads();
    if (threadIdx.x == 0) {
        tot = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); w += nwr) tot += red[w];
    }
    last_block_sum(tot, parts, counter, rr_out);
}

// max_r | |C(r)|^2 - 1 | of one coil map into *dev (non-negative float bits: atomicMax exact).
__global__ void __launch_bounds__(kThreads)
coil_unimodular_kernel(const float2* __restrict__ C, size_t npix, unsigned int* __restrict__ dev) {
    float m = 0.f;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < npix;
         i += (size_t)gridDim.x * blockDim.x) {
        const float2 v = C[i];
        m = fmaxf(m, fabsf(fmaf(v.x, v.x, v.y * v.y) - 1.f));
    }
    m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 16));
    m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 8));
    m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 4));
    m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 2));
    m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 1));
    if ((threadIdx.x & 31) == 0) atomicMax(dev, __float_as_uint(m));
}

// y = W_S x (no lambda); parity tests only.
template <int M>
__global__ void __launch_bounds__(kThreads)
apply_w_kernel(const float2* __restrict__ x, const float2* __restrict__ S, float2* __restrict__ y,
               int T, int circ, size_t npix) {
    const int k = circ ? T : T - M + 1;
    for (size_t px = (size_t)blockIdx.x * blockDim.x + threadIdx.x; px < npix;
         px += (size_t)gridDim.x * blockDim.x) {
        float2 s[M][M];
        load_S<M>(S, npix, px, s);
        for (int n = 0; n < T; ++n) {
            float2 w = make_float2(0.f, 0.f);
#pragma unroll
            for (int a = 0; a < M; ++a) {
                const int j = n - M + 1 + a;
                if (!circ && (j < 0 || j >= k)) continue;  // circ: every window
#pragma unroll
                for (int b = 0; b < M; ++b)
                    w = cfma(s[a][b], x[(size_t)wrap_frame(n + a - b, T) * npix + px], w);
            }
            y[(size_t)n * npix + px] = w;
        }
    }
}

// Grid of a row kernel: one CTA per row while the rows fit one resident wave, else one wave
// (the CTAs then loop over rows), so that the pass leaves at most a wave of partials.
// The occupancy query costs more host time than a launch: its answers are kept (a few shapes per
// kernel; the table is shared by all threads).
template <typename K>
cudaError_t row_grid(K kern, int threads, size_t smem, long long rows, int* grid) {
    static std::mutex mu;
    static std::map<std::tuple<int, const void*, int, size_t>, int> known;
    int dev = 0, per_sm = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const auto key = std::make_tuple(dev, reinterpret_cast<const void*>(kern), threads, smem);
    {
        std::lock_guard<std::mutex> lock(mu);
        auto it = known.find(key);
        if (it != known.end()) per_sm = it->second;
    }
    if (!per_sm) {
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, threads, smem);
        if (e != cudaSuccess) return e;
        if (per_sm < 1) return cudaErrorLaunchOutOfResources;  // no CTA of this shape fits an SM
        std::lock_guard<std::mutex> lock(mu);
        if (known.size() < 4096) known[key] = per_sm;
    }
    long long wave = (long long)per_sm * num_sms();
    if (wave > kMaxParts) wave = kMaxParts;
    *grid = (int)(rows < wave ? rows : wave);
    return cudaSuccess;
}

template <int N, int M>
cudaError_t launch_row_inv_w_NM(const Dims& d, const Twiddles& tw, float2* t, const float2* p,
                                const float2* S, float lam, Partials* pq, cudaStream_t st) {
    using F = RowFft<N>;
    const int rows = d.rows();
    int grid = 0;
    auto k = d.circ ? row_inv_w_kernel<F, N, M, true> : row_inv_w_kernel<F, N, M, false>;
    const RunShape v = run_shape<F, N, M>(d.T, rows);
    const size_t smem = ((size_t)v.bufs * F::kBuf + N) * sizeof(float2);
    if (smem > kDynSmemFree) {
        cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    cudaError_t e = row_grid(k, v.threads, smem, (long long)rows * v.nrun, &grid);
    if (e != cudaSuccess) return e;
    pq->n = grid;
    return launch_pdl(k, dim3(grid), dim3(v.threads), smem, st, t, p, S, lam, d.T, rows, v.nrun, v.per,
                      pq->parts, tw.twQ);
}

template <int N>
cudaError_t launch_row_inv_w_N(const Dims& d, const Twiddles& tw, float2* t, const float2* p,
                               const float2* S, float lam, Partials* pq, cudaStream_t st) {
    switch (d.M) {
        case 1: return launch_row_inv_w_NM<N, 1>(d, tw, t, p, S, lam, pq, st);
        case 2: return launch_row_inv_w_NM<N, 2>(d, tw, t, p, S, lam, pq, st);
        case 3: return launch_row_inv_w_NM<N, 3>(d, tw, t, p, S, lam, pq, st);
        case 4: return launch_row_inv_w_NM<N, 4>(d, tw, t, p, S, lam, pq, st);
        case 5: return launch_row_inv_w_NM<N, 5>(d, tw, t, p, S, lam, pq, st);
        case 6: return launch_row_inv_w_NM<N, 6>(d, tw, t, p, S, lam, pq, st);
        default: return cudaErrorInvalidValue;
    }
}

int pix_grid(size_t npix) {
    const size_t g = (npix + kThreads - 1) / kThreads;
    return (int)(g < (size_t)kMaxParts ? g : (size_t)kMaxParts);
}

// One resident wave: kUpdPerSM CTAs per SM (fewer for small problems), grid-stride inside.
int upd_grid(size_t n4) {
    const size_t per = (size_t)kUpdThreads * kUpdVec;
    const size_t need = (n4 + per - 1) / per;
    size_t g = (size_t)num_sms() * kUpdPerSM;
    if (need < g) g = need;
    return (int)(g < 1 ? 1 : (g < (size_t)kMaxParts ? g : (size_t)kMaxParts));
}

template <int N, int M, bool ADJ>
cudaError_t launch_coil_inv_NM(const Dims& d, const Twiddles& tw, float2* t, const float2* p,
                               const float2* coils, const float2* S, float lam, double* pq_parts,
                               float2* x_out, cudaStream_t st) {
    auto k = coil_row_inv_kernel<N, M, ADJ>;
    // (the series that the coil passes take: four copies of the rows within the shared memory)
    if (((size_t)4 * d.T * N + N) * sizeof(float2) > 220 * 1024) return cudaErrorInvalidValue;
    const InvShape v = inv_shape<N>(d.T);
    const size_t smem = ((size_t)v.bufs * RegFft<N>::kBuf + N) * sizeof(float2);
    if (smem > kDynSmemFree) {
        cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    return launch_pdl(k, dim3(d.P), dim3(v.threads), smem, st, t, p, coils, S, lam, d.T, d.P, d.nc,
                      v.passes, v.per, pq_parts, x_out, tw.twQ);
}

template <int N, bool ADJ>
cudaError_t launch_coil_inv_N(const Dims& d, const Twiddles& tw, float2* t, const float2* p,
                              const float2* coils, const float2* S, float lam, double* pq_parts,
                              float2* x_out, cudaStream_t st) {
    if constexpr (ADJ) {
        return launch_coil_inv_NM<N, 1, true>(d, tw, t, p, coils, S, lam, pq_parts, x_out, st);
    } else {
        switch (d.M) {
#define CASE(MM) \
    case MM: return launch_coil_inv_NM<N, MM, false>(d, tw, t, p, coils, S, lam, pq_parts, x_out, st);
            CASE(1) CASE(2) CASE(3) CASE(4) CASE(5) CASE(6)
#undef CASE
            default: return cudaErrorInvalidValue;
        }
    }
}

template <bool ADJ>
cudaError_t launch_coil_inv(const Dims& d, const Twiddles& tw, float2* t, const float2* p,
                            const float2* coils, const float2* S, float lam, double* pq_parts,
                            float2* x_out, cudaStream_t st) {
    if (d.P > kMaxParts) return cudaErrorInvalidValue;
    switch (d.Q) {
#define CASE(NN) \
    case NN: return launch_coil_inv_N<NN, ADJ>(d, tw, t, p, coils, S, lam, pq_parts, x_out, st);
        CASE(16) CASE(32) CASE(64) CASE(128) CASE(192) CASE(256) CASE(512)
#undef CASE
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace

int num_sms() {
    static int cache[64] = {0};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 132;
    if (!cache[dev]) {
        int n = 0;
        if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n < 1) n = 132;
        cache[dev] = n;
    }
    return cache[dev];
}

int w_max_M() { return kMaxM; }
int w_max_frames_times_q() { return (200 * 1024) / (3 * (int)sizeof(float2)); }
int max_parts() { return kMaxParts; }

cudaError_t launch_row_inv_w(const Dims& d, const Twiddles& tw, float2* t, const float2* p,
                             const float2* S, float lam, Partials* pq, cudaStream_t st) {
    switch (d.Q) {
        case 16: return launch_row_inv_w_N<16>(d, tw, t, p, S, lam, pq, st);
        case 32: return launch_row_inv_w_N<32>(d, tw, t, p, S, lam, pq, st);
        case 64: return launch_row_inv_w_N<64>(d, tw, t, p, S, lam, pq, st);
        case 128: return launch_row_inv_w_N<128>(d, tw, t, p, S, lam, pq, st);
        case 192: return launch_row_inv_w_N<192>(d, tw, t, p, S, lam, pq, st);
        case 256: return launch_row_inv_w_N<256>(d, tw, t, p, S, lam, pq, st);
        case 512: return launch_row_inv_w_N<512>(d, tw, t, p, S, lam, pq, st);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_coil_row_inv_w(const Dims& d, const Twiddles& tw, float2* t, const float2* p,
                                  const float2* coils, const float2* S, float lam, Partials* pq,
                                  cudaStream_t st) {
    pq->n = d.P;
    return launch_coil_inv<false>(d, tw, t, p, coils, S, lam, pq->parts, nullptr, st);
}

cudaError_t launch_coil_combine(const Dims& d, const Twiddles& tw, float2* t, const float2* coils,
                                float2* x, cudaStream_t st) {
    return launch_coil_inv<true>(d, tw, t, nullptr, coils, nullptr, 0.f, nullptr, x, st);
}

cudaError_t launch_cg_update(const Dims& d, float2* x, float2* r, const float2* p,
                             const float2* q, const double* rr_in, const Partials& pq,
                             Partials* rr, double* alpha, bool with_x, cudaStream_t st) {
    const size_t n4 = d.elems() / 2;  // two complex values per float4
    const int grid = upd_grid(n4);
    rr->n = grid;
    return launch_pdl(with_x ? cg_update_kernel<true> : cg_update_kernel<false>, dim3(grid),
                      dim3(kUpdThreads), 0, st, reinterpret_cast<float4*>(x),
                      reinterpret_cast<float4*>(r), reinterpret_cast<const float4*>(p),
                      reinterpret_cast<const float4*>(q), n4, rr_in, (const double*)pq.parts, pq.n,
                      rr->parts, alpha);
}

cudaError_t launch_sum_partials(const Partials& in, double* out, cudaStream_t st) {
    sum_partials_kernel<<<1, 32, 0, st>>>(in.parts, in.n, out);
    return cudaGetLastError();
}

// Frames of a run of the residual carry: the longest of 16, 8, 4, 2 (no longer than the series needs: the
// registers are those of the whole run) that leaves enough threads in flight, 2 for the smallest series:
// about ten warps an SM, and twenty for runs of 16 with up to four taps, whose weights are few to read
// again (256x256x16, M = 3: two runs 1.3 us less than one; M = 6: one run 4.2 us less than two;
// 256x512x5, M = 3: runs of 8 37 us a call, of 16 41).
int resid_run(const Dims& d) {
    int fc = 16;
    while (fc > 2 && fc / 2 >= d.T) fc /= 2;
    auto fill = [&] { return (long long)d.pixels() * ((d.T + fc - 1) / fc); };
    while (fc > 2 && fill() < (fc == 16 && d.M <= 4 ? 90000 : 50000)) fc /= 2;
    return fc;
}

cudaError_t launch_resid_carry(const Dims& d, float2* r, const float2* x, const float2* S_old,
                               const float2* S_new, float lam, int first, const RedSlot& rs,
                               double* rr_out, cudaStream_t st, const float2* aha_x) {
    const size_t npix = d.pixels();
    const int fc = resid_run(d), nrun = (d.T + fc - 1) / fc, run = (d.T + nrun - 1) / nrun;
    const int nwr = nrun < kResWarps ? nrun : kResWarps;   // warps of a pixel group
    const int ngrp = nwr >= 4 ? 1 : 4 / nwr;               // at least about four warps a CTA
    const size_t blocks = (npix / 32 + ngrp - 1) / ngrp;
    const dim3 grid((unsigned)(blocks < (size_t)kMaxParts ? blocks : (size_t)kMaxParts));
    const dim3 block(32 * nwr * ngrp);
    const size_t smem = nrun > 1 ? (size_t)ngrp * d.T * 32 * sizeof(float) : 0;
#define RUN(MM, FF)                                                                                 \
    {                                                                                               \
        auto kern = resid_carry_kernel<MM, FF>;                                                     \
        if (smem > kDynSmemFree) {                                                                  \
            cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, \
                                                 (int)smem);                                        \
            if (e != cudaSuccess) return e;                                                         \
        }                                                                                           \
        return launch_pdl(kern, grid, block, smem, st, r, x, aha_x, S_old, S_new, lam, first, d.T,  \
                          d.circ, npix, nrun, run, nwr, rs.parts, rs.counter, rr_out);              \
    }
#define CASE(MM)                       \
    case MM:                           \
        if (fc == 16) RUN(MM, 16)      \
        if (fc == 8) RUN(MM, 8)        \
        if (fc == 4) RUN(MM, 4)        \
        RUN(MM, 2)
    switch (d.M) {
        CASE(1) CASE(2) CASE(3) CASE(4) CASE(5) CASE(6)
        default: return cudaErrorInvalidValue;
    }
#undef CASE
#undef RUN
}

cudaError_t launch_coil_unimodular(const Dims& d, const float2* coils, unsigned int* dev,
                                   cudaStream_t st) {
    cudaError_t e = cudaMemsetAsync(dev, 0, sizeof(unsigned int), st);
    if (e != cudaSuccess) return e;
    coil_unimodular_kernel<<<pix_grid(d.pixels()), kThreads, 0, st>>>(coils, d.pixels(), dev);
    return cudaGetLastError();
}

cudaError_t launch_apply_w(const Dims& d, const float2* x, const float2* S, float2* y,
                           cudaStream_t st) {
    const int g = pix_grid(d.pixels());
#define CASE(MM)                                                                        \
    case MM: apply_w_kernel<MM><<<g, kThreads, 0, st>>>(x, S, y, d.T, d.circ, d.pixels()); break;
    switch (d.M) {
        CASE(1) CASE(2) CASE(3) CASE(4) CASE(5) CASE(6)
        default: return cudaErrorInvalidValue;
    }
#undef CASE
    return cudaGetLastError();
}

}  // namespace recon
