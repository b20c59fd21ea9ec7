// yline.cuh -- the Y pass with two radix stages and one exchange (lengths 125 to 1024).
//
// k_colpass_tma brings a tile of columns into shared memory, runs its radix stages there with a
// CTA barrier before and after each exchange, and stores the tile from shared memory: volumes
// that stay in L2 move at a third of its rate (256x256x128: 16.5 us per launch, 7 at the L2 copy
// rate).  Here N = R0 R1 with radices of up to 32: the first butterflies take their elements
// straight from global memory, the second ones store theirs straight back, and the tile passes
// through shared memory once, with one barrier.  The loads in flight (a thread's whole
// butterfly) and two to four CTAs per SM cover the latency.
//
// Forward and inverse together, best other launch shape -> this one (us), 48 planes of 129
// columns / 96 planes of 321: length 128 16.2 -> 14.6 / 26.5 -> 25.0; 160 18.1 -> 16.2 / 32.7 ->
// 30.3; 192 17 -> 16.4 / 37.2 -> 33.8; 256 20.4 -> 17.0 / 47.4 -> 42.2; 320 24.5 -> 20.4 / 68.5 -> 66.6;
// 384 26.4 -> 24.0 / 76.5 -> 81.6; 512 30.5 -> 28.6 / 104 -> 104; 640 45.0 -> 33.0 / 172 -> 145; 768 45.3
// -> 39 / 178 -> 165; 1024 55.5 -> 50.2 / 190 -> 228.  256x256x128, a whole RL run of 100: 11.5 ->
// 10.65 ms.  Lengths above 1024 (radices of 45 to 54, 6 warps per CTA, 4 columns) were 6 to 43%
// slower than the tile pipeline and are not built.
#pragma once

#include "line.cuh"

namespace cubic {

// smaller radix first, as near to a square as the length allows
constexpr int yline_r0(int N)
{
    int best = 0;
    for (int r = 2; r * r <= N; ++r)
        if (N % r == 0) best = r;
    return best;
}
template <int N>
using YLine = LineR<yline_r0(N), N / yline_r0(N)>;
constexpr bool yline_has(int N) { return N >= 125 && yline_r0(N) > 1 && N / yline_r0(N) <= 32; }
// Whether a plan that was not tuned takes it: at 1024, where the tile pipeline has two 64 KB stages, a
// volume larger than L2 is 20% slower with it (a smaller one 10% faster: the tuner's choice).
constexpr bool yline_default(int N) { return yline_has(N) && N <= 768; }
// The same for volumes past L2.  There the kernel's loads wait on HBM, and its advantage hangs on
// what runs beside it.  Plain call, us an iteration, tile pipeline / this kernel, with a real PSF
// spectrum: 384 (128 planes of 640 and 768, 100 of 1024) 504 / 537, 599 / 638, 624 / 675; 512 (128 of 512, 64 of
// 1024, 81 of 768) 533 / 553, 525 / 554, 501 / 521; 768 (100 of 512 and 768, 64 of 768) 684 / 705, 998 /
// 1051, 645 / 671.  With a complex one, which makes the Z pass the longer: 384 526 / 558, 627 / 668, 635 /
// 622; 512 558 / 577, 548 / 544, 514 / 504; 768 694 / 656, 1023 / 980, 677 / 641.  256 and 640 gain in
// either case (128 of 1024: 577 / 506; 90 of 768: 768 / 732).
constexpr bool yline_large(int N, bool real_h)
{
    return yline_default(N) && N != 512 && !(real_h && (N == 384 || N == 768));
}
// columns per CTA: 128-byte segments where they leave room for two CTAs per SM
constexpr int yline_cols(int N) { return N <= 320 || N == 512 ? 16 : 8; }
// first-stage butterflies per thread: with R1 = 2 R0 two of them hold what the second stage's does
template <int N>
constexpr int yline_first() { return YLine<N>::R1 == 2 * YLine<N>::R0 ? 2 : 1; }
template <int N>
constexpr int yline_threads() { return (YLine<N>::R1 / yline_first<N>() * yline_cols(N) + 31) / 32 * 32; }
// registers per thread by the larger radix
template <int N>
constexpr int yline_ctas()
{
    const int r = YLine<N>::R1, regs = r <= 16 ? 64 : r <= 20 ? 80 : r <= 24 ? 96 : 128;
    const int c = 65536 / (regs * yline_threads<N>());
    return c > 0 ? c : 1;
}
// a row of R1 positions takes an odd number of slots, so that the second stage's reads (one
// row per butterfly) spread over the banks
template <int N>
constexpr int yline_step() { return YLine<N>::R1 | 1; }
template <int N>
constexpr size_t yline_smem()
{
    return ((size_t)YLine<N>::R0 * yline_step<N>() * yline_cols(N) + YLine<N>::kTw) * sizeof(float2);
}

// Grid (column tiles, planes).  The inverse runs on conjugated data.
template <int N>
__global__ void __launch_bounds__(yline_threads<N>(), yline_ctas<N>()) k_yline(const __grid_constant__ YArgs a)
{
    using F = YLine<N>;
    constexpr int R0 = F::R0, R1 = F::R1, B = yline_cols(N), T = yline_threads<N>(), S = yline_step<N>();
    constexpr int Q = yline_first<N>(), P = R1 / Q;  // butterflies j and j + P of the first stage
    extern __shared__ __align__(16) float2 smem_yl[];
    float2 *tw = smem_yl + R0 * S * B;
    const int c = threadIdx.x % B, j = threadIdx.x / B;
    const int64_t col = a.col0 + (int64_t)blockIdx.x * B + c;
    const bool ok = col < a.col1;
    float2 *base = a.spec + (int64_t)blockIdx.y * N * a.xp + col;
    const float sg = a.inverse ? -1.f : 1.f;
    const int nl = a.nload > 0 ? (int)a.nload : N, ns = a.nstore > 0 ? (int)a.nstore : N;
    pdl_wait();
    pdl_trigger();
    float2 x[Q][R0];
    static_for<0, Q>([&](auto q_) {
        constexpr int q = CUBIC_CI(q_);
        const float2 *p = base + (int64_t)(j + q * P) * a.xp;
        static_for<0, R0>([&](auto r_) {
            constexpr int r = CUBIC_CI(r_);
            x[q][r] = make_float2(0.f, 0.f);
            if (ok && j < P && j + q * P + r * R1 < nl) x[q][r] = p[(int64_t)(r * R1) * a.xp];
        });
    });
    F::fill_twiddles(tw, a.tw, threadIdx.x, T);  // under the loads
    __syncthreads();
    if (j < P) {
        static_for<0, Q>([&](auto q_) {
            constexpr int q = CUBIC_CI(q_);
            static_for<0, R0>([&](auto r_) { x[q][CUBIC_CI(r_)].y *= sg; });
            F::fwd0(x[q], tw, j + q * P);
            static_for<0, R0>([&](auto r_) { smem_yl[(CUBIC_CI(r_) * S + j + q * P) * B + c] = x[q][CUBIC_CI(r_)]; });
        });
    }
    __syncthreads();
    if (j < R0) {
        float2 y[R1];
        static_for<0, R1>([&](auto r_) { y[CUBIC_CI(r_)] = smem_yl[(j * S + CUBIC_CI(r_)) * B + c]; });
        Dft<R1, kPacked>::run(y);
        float2 *p = base + (int64_t)j * a.xp;
        static_for<0, R1>([&](auto r_) {
            constexpr int r = CUBIC_CI(r_);
            if (ok && j + r * R0 < ns) p[(int64_t)(r * R0) * a.xp] = make_float2(y[r].x, sg * y[r].y);
        });
    }
}

}  // namespace cubic
