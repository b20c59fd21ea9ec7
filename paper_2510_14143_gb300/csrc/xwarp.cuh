// xwarp.cuh -- the X pass with one warp per group of line pairs (lengths 256 to 1024).
//
// k_xpass spreads a line pair over a CTA's worth of threads with at most 16 elements each:
// three radix stages, an exchange for the split into the two rows' spectra, and CTA barriers
// in between (about 4600 warp instructions per line pair at length 1024, which bound the ratio
// pass at 65% of the DRAM rate).  Here a pair lives in one warp and takes two stages
// (N = R0 R1, in place, see plane.cuh), with warp synchronisation only.  Frequency k and its
// partner N - k sit in lanes b and R0 - b at mirrored registers, so the split and the merge
// are shuffles instead of passes through shared memory, and the spectrum rows load and store
// in natural order straight from registers.  16 warps per SM (24 at length 256): a butterfly of
// up to 32 elements takes up to 128 registers.
//
// Ratio and update pass together, best other launch shape -> this one (us): 65536 lines of 1024
// (1024x1024x128 voxels) 763 -> 645; 8192 lines of 256 24.5 -> 20.1, of 320 32.7 -> 27.9, of 384
// 33.2 -> 28.6, of 512 36.6 -> 35.1, of 640 58.3 -> 44.1, of 768 60.4 -> 49.8, of 1024 63.7 ->
// 64.8.  The shapes that plans not tuned took before are further off (640: 93 us).
#pragma once

#include "line.cuh"

namespace cubic {

constexpr int kXWarps = 8;

// the line's radices: R0 x 16 up to 512, R0 x 32 from 640 (R0 = 16 to 32)
template <int N>
using XLine = LineR<N / (N > 512 ? 32 : 16), (N > 512 ? 32 : 16)>;
constexpr bool xwarp_has(int N)
{
    return N == 256 || N == 320 || N == 384 || N == 512 || N == 640 || N == 768 || N == 1024;
}
// line pairs of a warp: as many as fill the lanes
template <int N>
constexpr int xwarp_lines() { return 32 / XLine<N>::R1; }
template <int N>
constexpr size_t xwarp_smem()
{
    return ((size_t)XLine<N>::kTw + (size_t)kXWarps * xwarp_lines<N>() * XLine<N>::kSlots) * sizeof(float2);
}

__device__ __forceinline__ float2 shfl2(float2 v, int lane)
{
    return make_float2(__shfl_sync(0xffffffffu, v.x, lane), __shfl_sync(0xffffffffu, v.y, lane));
}

template <int N, int MODE>
__global__ void __launch_bounds__(kXWarps * 32, (N <= 256 ? 3 : 2)) k_xwarp(const __grid_constant__ XArgs a)
{
    using F = XLine<N>;
    constexpr int R0 = F::R0, R1 = F::R1, Lw = xwarp_lines<N>(), HK = R1 / 2;
    // second stage: LG lines side by side in a group of lanes, G groups one after the other
    constexpr int LG = 32 / R0, G = Lw / LG;
    static_assert(Lw * R1 == 32 && R0 <= 32 && LG * G == Lw, "a warp's lanes hold whole lines");
    extern __shared__ __align__(16) float2 smem_xw[];
    constexpr bool kIn = MODE != XM_FWD, kOut = MODE != XM_INV && MODE != XM_FINAL;
    float2 *tw = smem_xw;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    float2 *buf = smem_xw + F::kTw + warp * Lw * F::kSlots;
    const int64_t pair0 = ((int64_t)blockIdx.x * kXWarps + warp) * Lw;
    const int64_t pairs = (a.rows + 1) / 2;
    auto srow = [&](int64_t r) -> int64_t {
        if (a.ny_img <= 0) return r;
        const unsigned q = (unsigned)r / (unsigned)a.ny_img;
        return (int64_t)q * a.ny_spec + ((unsigned)r - q * (unsigned)a.ny_img);
    };
    if constexpr (MODE == XM_RATIO || MODE == XM_UPDATE || MODE == XM_FINAL) {
        // the warp's operand rows into L2 (a hint, so before the wait)
        const int64_t left = a.rows - 2 * pair0;
        if (lane == 0 && left > 0)
            bulk_prefetch_l2((MODE == XM_RATIO ? a.d : a.u) + pair0 * 2 * N,
                             (unsigned)((left < 2 * Lw ? left : 2 * Lw) * N * sizeof(float)));
    }
    F::fill_twiddles(tw, a.tw, threadIdx.x, kXWarps * 32);
    __syncthreads();
    pdl_wait();
    PointSums sum;

    // second-stage butterfly of group g: line l, index b; its values are frequencies b + R0 r
    const int lg = lane / R0, b = lane - lg * R0, mirror = lg * R0 + (b == 0 ? 0 : R0 - b);
    const bool in = lg < LG, zero = b == 0;
    if constexpr (kIn) {
        static_for<0, G>([&](auto g_) {
            const int l = CUBIC_CI(g_) * LG + lg;
            const int64_t pair = pair0 + l;
            const bool ok = in && pair < pairs, two = in && 2 * pair + 1 < a.rows;
            const float2 *q0 = a.spec_in + srow(2 * pair) * a.xp, *q1 = a.spec_in + srow(2 * pair + 1) * a.xp;
            float2 x[R1], w[HK];
            static_for<0, HK>([&](auto r_) {
                constexpr int r = CUBIC_CI(r_);
                float2 A = ok ? q0[b + R0 * r] : make_float2(0.f, 0.f), B = two ? q1[b + R0 * r] : make_float2(0.f, 0.f);
                if (r == 0 && zero) A.y = B.y = 0.f;  // real lines: self-conjugate bins
                // conjugated for the inverse: Z[k] = A + iB, Z[N - k] = conj A + i conj B
                x[r] = make_float2(A.x - B.y, -A.y - B.x);
                w[r] = make_float2(A.x + B.y, A.y - B.x);
            });
            const float2 ny = zero && ok ? make_float2(q0[N / 2].x, two ? -q1[N / 2].x : 0.f) : make_float2(0.f, 0.f);
            float2 next = ny;  // lane b = 0: the value of the register before
            static_for<0, HK>([&](auto u_) {
                constexpr int r = HK - 1 - CUBIC_CI(u_);
                const float2 got = shfl2(w[r], mirror);
                x[R1 - 1 - r] = zero ? next : got;
                next = got;
            });
            Dft<R1, kPacked>::run(x);
            if (in) {
                float2 *q = buf + l * F::kSlots + b * F::kStep;
                static_for<0, R1>([&](auto r_) { q[CUBIC_CI(r_)] = x[CUBIC_CI(r_)]; });
            }
        });
        __syncwarp();
    }
    {
        const int l = lane / R1, j = lane % R1;
        const int64_t pair = pair0 + l;
        float2 *q = buf + l * F::kSlots + j;
        float2 x[R0];
        if constexpr (kIn) {
            static_for<0, R0>([&](auto r_) { x[CUBIC_CI(r_)] = q[CUBIC_CI(r_) * F::kStep]; });
            F::bwd0(x, tw, j);
            static_for<0, R0>([&](auto r_) { x[CUBIC_CI(r_)].y = -x[CUBIC_CI(r_)].y; });
        }
        if (!kIn) static_for<0, R0>([&](auto r_) { x[CUBIC_CI(r_)] = make_float2(0.f, 0.f); });
        const int64_t o = 2 * pair * N + j;
        if (pair < pairs) plane_point<MODE, R0, R1>(a, x, o, o + N, 2 * pair + 1 < a.rows, sum, a.center);
        if constexpr (kOut) {
            F::fwd0(x, tw, j);
            static_for<0, R0>([&](auto r_) { q[CUBIC_CI(r_) * F::kStep] = x[CUBIC_CI(r_)]; });
        }
    }
    if constexpr (kOut) {
        __syncwarp();
        static_for<0, G>([&](auto g_) {
            const int l = CUBIC_CI(g_) * LG + lg;
            const int64_t pair = pair0 + l;
            const bool ok = in && pair < pairs, two = in && 2 * pair + 1 < a.rows;
            float2 *q0 = a.spec_out + srow(2 * pair) * a.xp, *q1 = a.spec_out + srow(2 * pair + 1) * a.xp;
            const float2 *q = buf + (in ? l * F::kSlots + b * F::kStep : 0);
            float2 x[R1];
            static_for<0, R1>([&](auto r_) { x[CUBIC_CI(r_)] = q[CUBIC_CI(r_)]; });
            Dft<R1, kPacked>::run(x);
            float2 before = x[0];  // lane b = 0: Z[N - R0 r] is the register before's partner
            static_for<0, HK>([&](auto r_) {
                constexpr int r = CUBIC_CI(r_);
                const float2 zk = x[r], got = shfl2(x[R1 - 1 - r], mirror);
                const float2 zn = zero ? before : got;
                before = got;
                if (ok) q0[b + R0 * r] = make_float2(0.5f * (zk.x + zn.x), 0.5f * (zk.y - zn.y));
                if (two) q1[b + R0 * r] = make_float2(0.5f * (zk.y + zn.y), 0.5f * (zn.x - zk.x));
            });
            if (zero && ok) q0[N / 2] = make_float2(x[HK].x, 0.f);
            if (zero && two) q1[N / 2] = make_float2(x[HK].y, 0.f);
        });
    }
    point_sums_finish<MODE>(a, sum, (int)blockIdx.x, smem_xw);
}

}  // namespace cubic
