// Stockham transforms with the elements in registers: the passes of fft_smem (schedule 0: the same
// radices, twiddles and operations, so the same bits), N / 8 threads per sequence, eight elements
// each. Shared memory only carries the exchange between two passes (fft_num_stages - 1 of them), and
// the first pass takes its input, the last one leaves its output, straight in registers:
//
//   before a pass thread i holds the elements i + m N/8 (m < 8) in u[m]. A radix-R pass has N / R
//   butterflies, 8 / R per thread: butterfly j = i + b N/8 takes j + t N/R = i + (b + t 8/R) N/8,
//   i.e. u[b + t 8/R]; the last pass leaves its result t of butterfly j at element j + t N/R, the
//   same slots. N = 192 = 8 * 8 * 3 ends with 64 radix-3 butterflies over 24 threads: thread i takes
//   j = i + 24 b (b < 3, j < 64) from shared memory and leaves element j + 64 t in u[3 b + t].
#pragma once

#include "common.cuh"

namespace recon {

template <int N>
struct RegFft {
    static constexpr int kLanes = N / 8;                      // threads per sequence
    static constexpr bool kOdd = (N % 3 == 0);
    static constexpr int kOut = kOdd ? 9 : 8;                 // register slots of the result
    static constexpr int kBuf = N + N / 8;                    // exchange buffer per sequence
    static constexpr bool kWarp = (32 % kLanes) == 0;         // a sequence lies within one warp

    // Element of the result in slot m of thread i; negative: the slot is empty.
    RECON_DEV static int out_at(int i, int m) {
        if constexpr (!kOdd) return i + m * kLanes;
        const int j = i + kLanes * (m / 3);
        return j < N / 3 ? j + (N / 3) * (m % 3) : -1;
    }
    // Position in the exchange buffer: one element of padding per eight keeps the radix-8 writes
    // (stride 8) off each other's banks.
    RECON_DEV static int at(int e) { return e + (e >> 3); }

    // The threads of a sequence meet (of the CTA where sequences straddle warps: every thread of
    // the CTA then runs the transform).
    RECON_DEV static void sync() {
        if constexpr (kWarp) __syncwarp();
        else __syncthreads();
    }

    // es: stride of the exchange buffer's elements (1 for rows, the columns of a tile otherwise,
    // whose threads always meet in __syncthreads).
    template <bool INV, bool CTA_SYNC, int P = 1>
    RECON_DEV static void run(float2 (&u)[kOut], float2* sx, int es, const float2* tw, int i) {
        constexpr int R = fft_radix_at(N, P);
        constexpr bool last = P * R == N;
        if constexpr (R == 3) {
            static_assert(last, "the radix-3 pass comes last");
            constexpr int step = N / (P * R);
#pragma unroll
            for (int b = 0; b < 3; ++b) {
                const int j = i + b * kLanes;
                if (j >= N / 3) continue;
                float2 v[3];
#pragma unroll
                for (int t = 0; t < 3; ++t) v[t] = sx[at(j + t * (N / 3)) * es];
#pragma unroll
                for (int t = 1; t < 3; ++t) {
                    float2 w = tw[t * (j % P) * step];
                    if (INV) w.y = -w.y;
                    v[t] = cmul(v[t], w);
                }
                SmallDFT<3, INV>::run(v);
#pragma unroll
                for (int t = 0; t < 3; ++t) u[3 * b + t] = v[t];
            }
        } else {
            constexpr int B = 8 / R;
#pragma unroll
            for (int b = 0; b < B; ++b) {
                const int j = i + b * kLanes, k = j % P;
                float2 v[R];
#pragma unroll
                for (int t = 0; t < R; ++t) v[t] = u[b + t * B];
                if constexpr (P > 1) {
                    constexpr int step = N / (P * R);
#pragma unroll
                    for (int t = 1; t < R; ++t) {
                        float2 w = tw[t * k * step];
                        if (INV) w.y = -w.y;
                        v[t] = cmul(v[t], w);
                    }
                }
                SmallDFT<R, INV>::run(v);
#pragma unroll
                for (int t = 0; t < R; ++t) {
                    if constexpr (last) u[b + t * B] = v[t];
                    else sx[at((j - k) * R + k + t * P) * es] = v[t];
                }
            }
            if constexpr (!last) {
                meet<CTA_SYNC>();
                if constexpr (fft_radix_at(N, P * R) != 3) {
#pragma unroll
                    for (int m = 0; m < 8; ++m) u[m] = sx[at(i + m * kLanes) * es];
                    if constexpr (P * R * fft_radix_at(N, P * R) != N) meet<CTA_SYNC>();  // written again
                }
                run<INV, CTA_SYNC, P * R>(u, sx, es, tw, i);
            }
        }
    }

   private:
    template <bool CTA_SYNC>
    RECON_DEV static void meet() {
        if constexpr (CTA_SYNC) __syncthreads();
        else sync();
    }
};

}  // namespace recon
