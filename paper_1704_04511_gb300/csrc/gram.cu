// Gram matrix of the lifted matrix without forming it (Sec. III-B, Eq. gram-matrix,
// Eq. block-expression-for-R and Eq. P-ij-modified).
//
// G[(l, a), (l', b)] = lag_ab[l - l'],  lag_ab[d] = sum_r q_ab(r) e^{-2 pi i (d1 r1/P + d2 r2/Q)},
// q_ab(r) = sum_{j<k} conj(x_{j+M-1-a}(r)) x_{j+M-1-b}(r),   0 <= a <= b < M.
//
// The paper reads these lags out of the FFT of each product image. Only the (2N1-1) x (2N2-1)
// lags around zero are used, so they are evaluated directly as a pruned separable DFT:
//   gram_rows_kernel: one CTA per image row r1: the pair products of the row (a sliding window
//                     over the frames, all pairs per column in registers) and their pruned
//                     length-Q DFT Y[pair][d2][r1] (FP32 products with compensated sums: each
//                     accumulation carries the rounding errors of its additions in a second
//                     float, through the window sums, the DFT terms and the warp tree, and the
//                     pair becomes one FP64 value);
//   gram_fill_kernel: one warp per lag pair (d1, -d1): the length-P direction
//                     sum_r1 Y[pair][d2][r1] w_P^(d1 r1) in FP64 (fixed order, deterministic), then
//                     the lags scattered over the (l, l') pairs they fill in G (column-major s x s
//                     complex128, both triangles).
// Volumes (depth R, N3 depth taps; lag_ab[d] also carries w_R^(d3 r3)): the row kernel runs over
// the R * P rows unchanged, then the length-P and length-R directions are separated:
//   gram_depth_kernel: Z[pair][d2][d1][r3] = sum_r1 Y[pair][d2][r3 P + r1] w_P^(d1 r1)  (FP64);
//   gram_fill3_kernel: one warp per 3-D lag: sum_r3 Z[..][r3] w_R^(d3 r3) (FP64), scattered over
//                      the tap pairs of G with column index ((m N3 + l3) N1 + l1) N2 + l2.
#include "common.cuh"
#include "kernels.h"

namespace recon {

namespace {

// Threads of the row kernel: 512 (its DFT outputs spread over 16 warps) while the window sums of
// all pairs fit in the registers that leaves; 256 for M >= 5 (15 or 21 compensated pairs).
__host__ __device__ constexpr int row_threads(int M) { return M >= 5 ? 256 : 512; }

// kLo = false (only where the low parts do not fit in shared memory: M = 6 with 512-point rows
// and more than 12 frames): each window sum is rounded once to FP32 (hi + lo) before the DFT,
// whose terms and tree stay compensated. kTab: the twiddles of every output lag d2 are laid out
// contiguously in c ([L2][Q], built once per CTA), so that the lanes of a warp read consecutive
// entries; otherwise lane c reads w^(d2 c mod Q) from the length-Q table (bank conflicts for
// even d2). The same values either way. kReal: a frame's product with itself is |x|^2, taken as real (the
// general product leaves the rounding of re im - im re in its imaginary part), and its Y(-d2) is the
// conjugate of Y(d2): a quarter of the products and of the DFT outputs less at M = 3, and these bound
// the kernel (29.7 -> 21.4 us at 256x256x16, 9x9x3, with the staging and the table free of divisions).
template <int M, bool kLo, bool kReal, bool kTab>
__global__ void __launch_bounds__(row_threads(M))
gram_rows_kernel(const float2* __restrict__ x, int T, int P, int Q, int N2, int circ,
                 const float2* __restrict__ twQ, double2* __restrict__ Y) {
    constexpr int NP = M * (M + 1) / 2;
    extern __shared__ float2 sm[];
    // circ: T windows with frame indices taken mod T (the fully circulant lifting)
    const int k = circ ? T : T - M + 1, L2 = 2 * N2 - 1;
    float2* xs = sm;                         // [T][Q] row r1 of every frame
    float2* qp = xs + (size_t)T * Q;         // [NP][Q] pair products (compensated sum, high part)
    float2* ql = qp + (size_t)NP * Q;        // [NP][Q] their low parts (kLo)
    float2* tw = ql + (kLo ? (size_t)NP * Q : 0);  // [Q]
    float2* dtab = tw + Q;                   // [L2][Q] (kTab)
    const int r1 = blockIdx.x;
    for (int i = threadIdx.x; i < Q; i += blockDim.x) tw[i] = twQ[i];
    // (no divisions: they took as long as the products)
    for (int n = threadIdx.x >> 5; n < T; n += row_threads(M) / 32)
        for (int c = threadIdx.x & 31; c < Q; c += 32) xs[n * Q + c] = x[((size_t)n * P + r1) * Q + c];
    __syncthreads();
    if constexpr (kTab) {  // from the shared copy of the table (no further global loads)
        const int d2m0 = (Q - (N2 - 1) % Q) % Q;  // (-(N2 - 1)) mod Q; d2m0, c < Q <= 512
        for (int c = threadIdx.x; c < Q; c += blockDim.x) {
            int ti = (d2m0 * c) % Q;
            for (int i2 = 0; i2 < L2; ++i2) {
                dtab[i2 * Q + c] = tw[ti];
                ti += c;
                if (ti >= Q) ti -= Q;
            }
        }
    }
    // q_ab(c) = sum_j conj(x_{j+M-1-a}(c)) x_{j+M-1-b}(c): window w[m] = x_{j+M-1-m}(c)
    for (int c = threadIdx.x; c < Q; c += blockDim.x) {
        float2 w[M], acc[NP], lo[NP];
#pragma unroll
        for (int e = 0; e < NP; ++e) acc[e] = lo[e] = make_float2(0.f, 0.f);
#pragma unroll
        for (int m = 1; m < M; ++m) w[m] = xs[(M - 1 - m) * Q + c];
        for (int j = 0; j < k; ++j) {
            w[0] = xs[wrap_frame(j + M - 1, T) * Q + c];
            int e = 0;
#pragma unroll
            for (int a = 0; a < M; ++a)
#pragma unroll
                for (int b = a; b < M; ++b, ++e) {
                    const float2 t = cmulcj(w[a], w[b]);
                    comp_add(acc[e].x, lo[e].x, t.x);
                    if (!kReal || a != b) comp_add(acc[e].y, lo[e].y, t.y);
                }
#pragma unroll
            for (int m = M - 1; m > 0; --m) w[m] = w[m - 1];
        }
#pragma unroll
        for (int e = 0; e < NP; ++e) {
            if (kLo) {
                qp[e * Q + c] = acc[e];
                ql[e * Q + c] = lo[e];
            } else {
                qp[e * Q + c] = make_float2(__fadd_rn(acc[e].x, lo[e].x), __fadd_rn(acc[e].y, lo[e].y));
            }
        }
    }
    __syncthreads();
    // Y[pair][d2] = sum_c q[pair][c] w_Q^(d2 c); one warp per output, lanes stride c, each term
    // (hi + lo) w added to a compensated (hi, lo) pair, then a TwoSum shuffle tree
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // kReal: the pairs a < b with every d2 first, then the frames with themselves, d2 >= 0
    constexpr int NC = NP - M;
    const int nout = kReal ? NC * L2 + M * N2 : NP * L2;
    for (int o = warp; o < nout; o += row_threads(M) / 32) {
        int pr = o / L2, i2 = o % L2;
        bool self = false;
        if (kReal) {
            int a = 0;
            if (o < NC * L2) {  // the pr-th pair a < b
                int k = pr;
                while (k >= M - 1 - a) { k -= M - 1 - a; ++a; }
                pr = a * (2 * M - a + 1) / 2 + 1 + k;
            } else {
                self = true;
                a = (o - NC * L2) / N2;
                i2 = N2 - 1 + (o - NC * L2) % N2;
                pr = a * (2 * M - a + 1) / 2;
            }
        }
        const int d2m = (i2 - (N2 - 1) + Q) % Q;
        const float2* qrow = qp + (size_t)pr * Q;
        const float2* qlow = ql + (size_t)pr * Q;
        const float2* trow = dtab + (size_t)i2 * Q;
        int idx = (d2m * lane) % Q;
        const int step = (d2m * 32) % Q;
        float2 y = make_float2(0.f, 0.f), yl = make_float2(0.f, 0.f);
        if (kReal && self) {
#pragma unroll 4
            for (int c = lane; c < Q; c += 32) {
                const float2 wt = kTab ? trow[c] : tw[idx];
                const float q = qrow[c].x;
                comp_add(y.x, yl.x, __fmul_rn(q, wt.x));
                comp_add(y.y, yl.y, __fmul_rn(q, wt.y));
                if (kLo) {
                    const float l = qlow[c].x;
                    yl.x = __fadd_rn(yl.x, __fmul_rn(l, wt.x));
                    yl.y = __fadd_rn(yl.y, __fmul_rn(l, wt.y));
                }
                idx += step;
                if (idx >= Q) idx -= Q;
            }
        }
#pragma unroll 4
        for (int c = kReal && self ? Q : lane; c < Q; c += 32) {
            const float2 wt = kTab ? trow[c] : tw[idx];
            const float2 t = cmul(qrow[c], wt);
            comp_add(y.x, yl.x, t.x);
            comp_add(y.y, yl.y, t.y);
            if (kLo) {
                const float2 tl = cmul(qlow[c], wt);
                yl.x = __fadd_rn(yl.x, tl.x);
                yl.y = __fadd_rn(yl.y, tl.y);
            }
            idx += step;
            if (idx >= Q) idx -= Q;
        }
        // both components in one tree: lanes 0-15 take the real part, 16-31 the imaginary one
        const bool up = lane & 16;
        float h = up ? y.y : y.x, l = up ? yl.y : yl.x;
        float oh = __shfl_xor_sync(0xffffffffu, up ? y.x : y.y, 16);
        float ol = __shfl_xor_sync(0xffffffffu, up ? yl.x : yl.y, 16);
#pragma unroll
        for (int off = 8;; off >>= 1) {
            float sm_, er;
            two_sum(h, oh, sm_, er);
            h = sm_;
            l = __fadd_rn(__fadd_rn(l, ol), er);
            if (off == 0) break;
            oh = __shfl_xor_sync(0xffffffffu, h, off);
            ol = __shfl_xor_sync(0xffffffffu, l, off);
        }
        oh = __shfl_sync(0xffffffffu, h, 16);
        ol = __shfl_sync(0xffffffffu, l, 16);
        if (lane == 0) {
            const double2 z = make_double2((double)h + (double)l, (double)oh + (double)ol);
            Y[((size_t)pr * L2 + i2) * P + r1] = z;
            if (kReal && self) Y[((size_t)pr * L2 + (L2 - 1 - i2)) * P + r1] = zconj(z);
        }
    }
}

// One warp per lag (pair, d1, d2): the length-P direction in FP64 (lanes over r1 in a fixed
// order, then a fixed shuffle tree), then the lag scattered over the (l, l') pairs of G.
__global__ void gram_fill_kernel(const double2* __restrict__ Y, int P, int N1, int N2, int M,
                                 const double2* __restrict__ twPd, double2* __restrict__ lags,
                                 double2* __restrict__ G) {
    const int L1 = 2 * N1 - 1, L2 = 2 * N2 - 1, npair = M * (M + 1) / 2;
    const int nlag = npair * L1 * L2;
    const int s = N1 * N2 * M;
    const int o = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (o >= nlag) return;
    const int pr = o / (L1 * L2), rem = o % (L1 * L2);
    const int i1 = rem / L2, i2 = rem % L2;
    const int d1 = i1 - (N1 - 1), d2 = i2 - (N2 - 1);
    const int d1m = (d1 + P) % P;
    int a = 0, e = pr;
    while (e >= M - a) { e -= M - a; ++a; }
    const int b = a + e;
    // a frame with itself: lag_aa[-d] = conj(lag_aa[d]) exactly, so the warp of the lag in the
    // non-negative half (d1 > 0, or d1 = 0 and d2 >= 0) writes both and G is exactly Hermitian
    const bool self = a == b;
    if (self && (d1 < 0 || (d1 == 0 && d2 < 0))) return;
    const double2* yrow = Y + ((size_t)pr * L2 + i2) * P;
    double2 v = make_double2(0.0, 0.0);
    for (int r1 = lane; r1 < P; r1 += 32) v = zfma(yrow[r1], twPd[(d1m * r1) % P], v);
    v.x = warp_sum(v.x);
    v.y = warp_sum(v.y);
    if (self && d1 == 0 && d2 == 0) v.y = 0.0;  // sum of |x|^2
    if (lags && lane == 0) {
        lags[o] = v;
        if (self) lags[(size_t)pr * L1 * L2 + (size_t)(L1 - 1 - i1) * L2 + (L2 - 1 - i2)] = zconj(v);
    }
    const int lo1 = max(0, -d1), hi1 = min(N1, N1 - d1);
    const int lo2 = max(0, -d2), hi2 = min(N2, N2 - d2);
    const int n2 = hi2 - lo2, cnt = (hi1 - lo1) * n2;
    for (int t = lane; t < cnt; t += 32) {
        const int lp1 = lo1 + t / n2, lp2 = lo2 + t % n2;
        const int l1 = lp1 + d1, l2 = lp2 + d2;
        const size_t i = ((size_t)a * N1 + l1) * N2 + l2;
        const size_t j = ((size_t)b * N1 + lp1) * N2 + lp2;
        G[i + j * s] = v;
        if (i != j) G[j + i * s] = zconj(v);
    }
}

// The same with one warp per (pair, d1 >= 0, d2) for d1 and -d1 together (kReal series), rows r1 and
// P - r1 folded: with U = Y_r1 + Y_{P-r1} and V = Y_r1 - Y_{P-r1}, lag(+-d1) = sum U cos -+ i sum V sin (about
// a third of the FP64 operations of one warp per lag, on
// a pipe that issues one per 64 cycles and scheduler: 9.2 -> 7.1 us at 256x256x16, 9x9x3), lanes over
// r1 in a fixed order, then a fixed shuffle tree; then both lags scattered over the (l, l') pairs of G.
__global__ void gram_fill_pair_kernel(const double2* __restrict__ Y, int P, int N1, int N2, int M,
                                 const double2* __restrict__ twPd, double2* __restrict__ lags,
                                 double2* __restrict__ G) {
    const int L1 = 2 * N1 - 1, L2 = 2 * N2 - 1, npair = M * (M + 1) / 2;
    const int s = N1 * N2 * M;
    const int o = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (o >= npair * N1 * L2) return;
    const int pr = o / (N1 * L2), rem = o % (N1 * L2);
    const int d1 = rem / L2, i2 = rem % L2, d2 = i2 - (N2 - 1);
    int a = 0, e = pr;
    while (e >= M - a) { e -= M - a; ++a; }
    const int b = a + e;
    // a frame with itself: lag_aa[-d] = conj(lag_aa[d]) exactly, so the lag in the non-negative half
    // (d1 > 0, or d1 = 0 and d2 >= 0) gives both and G is exactly Hermitian
    const bool self = a == b;
    if (self && d1 == 0 && d2 < 0) return;
    const double2* yrow = Y + ((size_t)pr * L2 + i2) * P;
    const int H = P / 2;
    double2 E = make_double2(0.0, 0.0), O = E;
#pragma unroll 4
    for (int r1 = lane; r1 < H; r1 += 32) {
        const double2 w = twPd[(d1 * r1) % P];  // cos, -sin
        double2 u = yrow[r1];
        if (r1) {
            const double2 v = yrow[P - r1];
            O.x = fma(u.x - v.x, -w.y, O.x);
            O.y = fma(u.y - v.y, -w.y, O.y);
            u = zadd(u, v);
        }
        E.x = fma(u.x, w.x, E.x);
        E.y = fma(u.y, w.x, E.y);
    }
    if (lane == 0) {  // row P / 2
        const double2 u = yrow[H];
        E = (d1 & 1) ? make_double2(E.x - u.x, E.y - u.y) : zadd(E, u);
    }
    // the four sums in one tree: lane 8 k returns sum k of (E.x, E.y, O.x, O.y)
    const bool up = lane & 16, up8 = lane & 8;
    double p0 = up ? O.x : E.x, p1 = up ? O.y : E.y;
    p0 += __shfl_xor_sync(0xffffffffu, up ? E.x : O.x, 16);
    p1 += __shfl_xor_sync(0xffffffffu, up ? E.y : O.y, 16);
    double z = up8 ? p1 : p0;
    z += __shfl_xor_sync(0xffffffffu, up8 ? p0 : p1, 8);
#pragma unroll
    for (int off = 4; off > 0; off >>= 1) z += __shfl_xor_sync(0xffffffffu, z, off);
    E = make_double2(__shfl_sync(0xffffffffu, z, 0), __shfl_sync(0xffffffffu, z, 8));
    O = make_double2(__shfl_sync(0xffffffffu, z, 16), __shfl_sync(0xffffffffu, z, 24));
    // lag(+-d1) = E -+ i O; lanes 0-15 scatter d1, lanes 16-31 -d1 (a frame with itself: d1 alone)
    const bool neg = up && !self;
    double2 v = neg ? make_double2(E.x - O.y, E.y + O.x) : make_double2(E.x + O.y, E.y - O.x);
    if (d1 == 0) v = E;
    if (self && d1 == 0 && d2 == 0) v.y = 0.0;  // sum of |x|^2
    const int e1 = neg ? -d1 : d1;
    if (lags && (lane == 0 || (lane == 16 && neg && d1))) {
        double2* lp = lags + (size_t)pr * L1 * L2;
        lp[(size_t)(e1 + N1 - 1) * L2 + i2] = v;
        if (self) lp[(size_t)(N1 - 1 - d1) * L2 + (L2 - 1 - i2)] = zconj(v);
    }
    const int lo1 = max(0, -e1), hi1 = min(N1, N1 - e1);
    const int lo2 = max(0, -d2), hi2 = min(N2, N2 - d2);
    const int n2 = hi2 - lo2, cnt = (hi1 - lo1) * n2;
    const bool halves = !self && d1 != 0;  // 16 lanes per lag, else all 32
    for (int t = halves ? (lane & 15) : lane; t < cnt; t += halves ? 16 : 32) {
        const int lp1 = lo1 + t / n2, lp2 = lo2 + t % n2;
        const int l1 = lp1 + e1, l2 = lp2 + d2;
        const size_t i = ((size_t)a * N1 + l1) * N2 + l2;
        const size_t j = ((size_t)b * N1 + lp1) * N2 + lp2;
        G[i + j * s] = v;
        if (i != j) G[j + i * s] = zconj(v);
    }
}

// One warp per (pair, d2, d1, r3): the length-P direction of depth slice r3 (FP64, lanes over r1
// in a fixed order, then a fixed shuffle tree).
__global__ void gram_depth_kernel(const double2* __restrict__ Y, int P, int R, int N1, int N2,
                                  int npair, const double2* __restrict__ twPd,
                                  double2* __restrict__ Z) {
    const int L1 = 2 * N1 - 1, L2 = 2 * N2 - 1;
    const long long nout = (long long)npair * L2 * L1 * R;
    const long long o = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (o >= nout) return;
    const int r3 = (int)(o % R);
    const long long q = o / R;  // (pair * L2 + i2) * L1 + i1
    const int i1 = (int)(q % L1);
    const long long pi2 = q / L1;  // pair * L2 + i2
    const int d1m = ((i1 - (N1 - 1)) % P + P) % P;
    const double2* yrow = Y + (size_t)pi2 * R * P + (size_t)r3 * P;
    double2 v = make_double2(0.0, 0.0);
    for (int r1 = lane; r1 < P; r1 += 32) v = zfma(yrow[r1], twPd[(d1m * r1) % P], v);
    v.x = warp_sum(v.x);
    v.y = warp_sum(v.y);
    if (lane == 0) Z[o] = v;
}

// One warp per 3-D lag (pair, d3, d1, d2): the length-R direction in FP64, then the lag
// scattered over the tap pairs (l, l') with l - l' = d that it fills in G.
__global__ void gram_fill3_kernel(const double2* __restrict__ Z, int R, int N1, int N2, int N3,
                                  int M, const double2* __restrict__ twRd,
                                  double2* __restrict__ lags, double2* __restrict__ G) {
    const int L1 = 2 * N1 - 1, L2 = 2 * N2 - 1, L3 = 2 * N3 - 1, npair = M * (M + 1) / 2;
    const int nlag = npair * L3 * L1 * L2;
    const int s = N1 * N2 * N3 * M;
    const int o = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (o >= nlag) return;
    const int i2 = o % L2, i1 = (o / L2) % L1, i3 = (o / (L2 * L1)) % L3, pr = o / (L2 * L1 * L3);
    const int d1 = i1 - (N1 - 1), d2 = i2 - (N2 - 1), d3 = i3 - (N3 - 1);
    const int d3m = (d3 % R + R) % R;
    int a = 0, e = pr;
    while (e >= M - a) { e -= M - a; ++a; }
    const int b = a + e;
    // a frame with itself: only the non-negative half of the lags (d3 > 0, or d3 = 0 and
    // (d1, d2) non-negative as in 2-D) is summed; it writes the mirrored lag as its conjugate
    const bool self = a == b;
    if (self && (d3 < 0 || (d3 == 0 && (d1 < 0 || (d1 == 0 && d2 < 0))))) return;
    const double2* zrow = Z + (((size_t)pr * L2 + i2) * L1 + i1) * R;
    double2 v = make_double2(0.0, 0.0);
    for (int r3 = lane; r3 < R; r3 += 32) v = zfma(zrow[r3], twRd[(d3m * r3) % R], v);
    v.x = warp_sum(v.x);
    v.y = warp_sum(v.y);
    if (self && d3 == 0 && d1 == 0 && d2 == 0) v.y = 0.0;
    if (lags && lane == 0) {
        lags[o] = v;
        if (self)
            lags[(((size_t)pr * L3 + (L3 - 1 - i3)) * L1 + (L1 - 1 - i1)) * L2 + (L2 - 1 - i2)] = zconj(v);
    }
    const int lo1 = max(0, -d1), hi1 = min(N1, N1 - d1);
    const int lo2 = max(0, -d2), hi2 = min(N2, N2 - d2);
    const int lo3 = max(0, -d3), hi3 = min(N3, N3 - d3);
    const int n1 = hi1 - lo1, n2 = hi2 - lo2, cnt = (hi3 - lo3) * n1 * n2;
    for (int t = lane; t < cnt; t += 32) {
        const int lp2 = lo2 + t % n2, lp1 = lo1 + (t / n2) % n1, lp3 = lo3 + t / (n2 * n1);
        const size_t i = (((size_t)a * N3 + lp3 + d3) * N1 + lp1 + d1) * N2 + lp2 + d2;
        const size_t j = (((size_t)b * N3 + lp3) * N1 + lp1) * N2 + lp2;
        G[i + j * s] = v;
        if (i != j) G[j + i * s] = zconj(v);
    }
}

constexpr size_t kGramSmemMax = 220 * 1024;

size_t gram_smem_cfg(const Dims& d, bool lo, bool tab) {
    return ((size_t)d.T * d.Q + (lo ? 2 : 1) * (size_t)d.npair() * d.Q + d.Q +
            (tab ? (size_t)d.L2() * d.Q : 0)) * sizeof(float2);
}

// The shared-memory layout of the row kernel: the low parts first (accuracy), then the twiddle
// rows (speed), each where it fits.
void gram_cfg(const Dims& d, bool* lo, bool* tab) {
    *lo = gram_smem_cfg(d, true, false) <= kGramSmemMax;
    *tab = gram_smem_cfg(d, *lo, true) <= kGramSmemMax;
}

// Image series with rows of 64 and more elements: kReal (see gram_rows_kernel). Shorter rows are
// latency-bound either way, and volumes keep the last bits (their solves amplify those of S).
bool gram_real(const Dims& d) { return d.R == 1 && d.Q >= 64; }

}  // namespace

size_t gram_smem(const Dims& d) {
    bool lo, tab;
    gram_cfg(d, &lo, &tab);
    return gram_smem_cfg(d, lo, tab);
}

// One CTA per image row; the scratch holds the row DFTs Y[pair][d2][row] (complex128) and, for
// volumes, the depth-slice sums Z[pair][d2][d1][r3] after them.
int gram_blocks(const Dims& d) { return d.rows(); }

size_t gram_scratch_bytes(const Dims& d, int nblocks) {
    size_t b = (size_t)nblocks * d.npair() * d.L2() * sizeof(double2);
    if (d.R > 1) b += (size_t)d.npair() * d.L2() * d.L1() * d.R * sizeof(double2);
    return b;
}

cudaError_t launch_gram(const Dims& d, const Twiddles& tw, const float2* x, double2* lag_part,
                        int nblocks, double2* lags, double2* G, cudaStream_t st) {
    if (nblocks != d.rows()) return cudaErrorInvalidValue;
    const size_t smem = gram_smem(d);
    if (smem > kGramSmemMax) return cudaErrorInvalidValue;
    bool lo, tab;
    gram_cfg(d, &lo, &tab);
#define CASE(MM)                                                                                 \
    case MM: {                                                                                   \
        auto k = !lo ? (tab ? gram_rows_kernel<MM, false, false, true>                           \
                            : gram_rows_kernel<MM, false, false, false>)                         \
                 : gram_real(d) ? (tab ? gram_rows_kernel<MM, true, true, true>                  \
                                       : gram_rows_kernel<MM, true, true, false>)                \
                                : (tab ? gram_rows_kernel<MM, true, false, true>                 \
                                       : gram_rows_kernel<MM, true, false, false>);              \
        cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize,     \
                                             (int)smem);                                         \
        if (e != cudaSuccess) return e;                                                          \
        k<<<d.rows(), row_threads(MM), smem, st>>>(x, d.T, d.rows(), d.Q, d.N2, d.circ,           \
                                               tw.twQ, lag_part);                                \
        break;                                                                                   \
    }
    switch (d.M) {
        CASE(1) CASE(2) CASE(3) CASE(4) CASE(5) CASE(6)
        default: return cudaErrorInvalidValue;
    }
#undef CASE
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    if (d.R > 1) {
        double2* Z = lag_part + (size_t)nblocks * d.npair() * d.L2();
        const long long nz = (long long)d.npair() * d.L2() * d.L1() * d.R;
        gram_depth_kernel<<<(unsigned)((nz + 7) / 8), 256, 0, st>>>(lag_part, d.P, d.R, d.N1, d.N2,
                                                                    d.npair(), tw.twPd, Z);
        e = cudaGetLastError();
        if (e != cudaSuccess) return e;
        const int nlag3 = (int)d.nlag();
        gram_fill3_kernel<<<(nlag3 + 7) / 8, 256, 0, st>>>(Z, d.R, d.N1, d.N2, d.N3, d.M, tw.twRd,
                                                           lags, G);
        return cudaGetLastError();
    }
    if (gram_real(d)) {
        const int n = d.npair() * d.N1 * d.L2();
        gram_fill_pair_kernel<<<(n + 7) / 8, 256, 0, st>>>(lag_part, d.P, d.N1, d.N2, d.M, tw.twPd, lags, G);
        return cudaGetLastError();
    }
    const int nlag = d.npair() * d.L1() * d.L2();
    gram_fill_kernel<<<(nlag + 7) / 8, 256, 0, st>>>(lag_part, d.P, d.N1, d.N2, d.M, tw.twPd, lags, G);
    return cudaGetLastError();
}

}  // namespace recon
