// line.cuh -- lines of length N = R0 R1 in two in-place radix stages, and the pointwise
// Richardson-Lucy step on a thread's elements: what the plane kernels (plane.cuh) and the
// warp-per-line X kernels (xwarp.cuh) share.
//
// Decimation in frequency forward, decimation in time back: a line's frequencies stand in
// digit-reversed order (position k1 R1 + k2 holds frequency k1 + R0 k2), each thread rewrites
// the positions it read, and an exchange needs one synchronisation.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "passes.cuh"

namespace cubic {

// packed complex additions in the butterflies: 1 to 5% of an iteration (256x64x256 voxels
// 74.4 to 70.3 us, 100x100x100 44.0 to 42.9 us)
constexpr bool kPacked = true;

// N = R0 R1 with the smaller larger radix; R0 even for an even N (the c axis pairs element
// r with r + R0/2), R0 >= R1 where that leaves a choice, and R0 <= 16 (the pointwise step
// holds R0 elements: 125 = 5 x 25).
constexpr int plane_r0(int N)
{
    int best = 0, cost = 1 << 30;
    for (int r = 2; r < N; ++r) {
        if (N % r || (N % 2 == 0 && r % 2)) continue;
        const int q = N / r, c = 2 * (r > q ? r : q) + (r < q) + (r > 16 ? 64 : 0);
        if (c < cost) {
            cost = c;
            best = r;
        }
    }
    return best;
}
constexpr int plane_r1(int N) { return N / plane_r0(N); }

// Share of the lanes that work when a warp runs w lines of length N, both stages weighted by
// their elements, in percent
constexpr int warp_fill(int N, int w)
{
    const int a = plane_r0(N), b = plane_r1(N);
    return 200 * w * N / (32 * ((w * b + 31) / 32 * a + (w * a + 31) / 32 * b));
}

// Lines per warp task.  x lines: the fewest that fill 80% of the lanes (else the best of up
// to 8); c and p lines: 4, 8 or 16 adjacent ones (32-byte segments and up).
constexpr int row_lines(int N)
{
    int best = 1;
    for (int w = 1; w <= 8; ++w) {
        if (warp_fill(N, w) >= 80) return w;
        if (warp_fill(N, w) > warp_fill(N, best)) best = w;
    }
    return best;
}
constexpr int col_lines(int N)
{
    int best = 4;
    for (int w = 4; w <= 16; w *= 2) {
        if (warp_fill(N, w) >= 80) return w;
        if (warp_fill(N, w) > warp_fill(N, best)) best = w;
    }
    return best;
}

// p lines: 4 where they fill 70% of the lanes (the most warps, and a tile of at most 5 KB of
// shared memory each, so that 28 fit an SM), else 8
constexpr int conv_lines(int N) { return N > 40 && warp_fill(N, 4) >= 70 ? 4 : 8; }

template <int A, int B>
struct LineR {
    static constexpr int R0 = A, R1 = B;
    static constexpr int kTw = (R0 - 1) * R1;  // W_N^(j k) at [k - 1][j]
    // a line in shared memory: position p at slot p + p / R1 where R1 is even from 4 up, so
    // that the second stage's reads (stride R1 between threads) spread over the banks
    static constexpr int kStep = R1 + (R1 % 2 == 0 && R1 >= 4);
    static constexpr int kSlots = R0 * kStep;
    __host__ __device__ static constexpr int slot(int pos) { return pos / R1 * kStep + pos % R1; }
    __host__ __device__ static constexpr int pos_of(int q) { return q % R0 * R1 + q / R0; }
    __host__ __device__ static constexpr int freq_of(int pos) { return pos / R1 + R0 * (pos % R1); }

    // first stage forward, butterfly j: elements j + r R1 in, position r R1 + j out
    __device__ __forceinline__ static void fwd0(float2 (&x)[R0], const float2 *tw, int j)
    {
        Dft<R0, kPacked>::run(x);
        static_for<1, R0>([&](auto k_) { x[CUBIC_CI(k_)] = cmul(x[CUBIC_CI(k_)], tw[(CUBIC_CI(k_) - 1) * R1 + j]); });
    }
    // its mirror image, on conjugated data: the last stage of the inverse
    __device__ __forceinline__ static void bwd0(float2 (&x)[R0], const float2 *tw, int j)
    {
        static_for<1, R0>([&](auto k_) { x[CUBIC_CI(k_)] = cmul(x[CUBIC_CI(k_)], tw[(CUBIC_CI(k_) - 1) * R1 + j]); });
        Dft<R0, kPacked>::run(x);
    }
    __device__ __forceinline__ static void fill_twiddles(float2 *tw, const float2 *__restrict__ w, int tid, int n)
    {
        for (int i = tid; i < kTw; i += n) tw[i] = __ldg(w + (1 + i / R1) * (i % R1));
    }
};

template <int N>
using Line = LineR<plane_r0(N), plane_r1(N)>;

// ------------------------------------------------------------------ pointwise step

// What the pointwise step accumulates over a thread's lines
struct PointSums {
    float num = 0.f, den = 0.f;             // XM_UPDATE / XM_FINAL statistics
    CFloat nll{0.f, 0.f};                   // XM_RATIO likelihood
    CFloat acc_num{0.f, 0.f}, acc_den{0.f, 0.f};  // accelerated RL
};

// The pointwise step: v[i].x is element o0 + P i of the real volumes, v[i].y element o1 + P i
// (two: that row exists).  center: the pair at XArgs::center, or a
// copy of it in shared memory (null: none; k_xwarp passes the argument's, always null there, and
// not a literal: without the branches the ratio kernel at 256 measured 10% slower).
template <int MODE, int E, int P, class Off>
__device__ __forceinline__ void plane_point(const XArgs &a, float2 (&v)[E], const Off o0, const Off o1,
                                            const bool two, PointSums &sum, const float2 *center)
{
    if constexpr (MODE == XM_FWD) {
        const float *s0 = a.src + o0, *s1 = a.src + o1;
        if (a.acc_prev) {
            const float al = *a.acc_alpha;
            const float *p0 = a.acc_prev + o0, *p1 = a.acc_prev + o1;
            static_for<0, E>([&](auto i_) {
                constexpr int i = CUBIC_CI(i_);
                const int n = P * i;
                const float x0 = __ldg(s0 + n), x1 = two ? __ldg(s1 + n) : 0.f;
                const float q0 = __ldg(p0 + n), q1 = two ? __ldg(p1 + n) : 0.f;
                v[i] = make_float2(fmaxf(fmaf(al, x0 - q0, x0), 0.f), fmaxf(fmaf(al, x1 - q1, x1), 0.f));
            });
            float *y0 = a.acc_y + o0, *y1 = a.acc_y + o1;
            static_for<0, E>([&](auto i_) {
                constexpr int i = CUBIC_CI(i_);
                y0[P * i] = v[i].x;
                if (two) y1[P * i] = v[i].y;
            });
        } else {
            static_for<0, E>([&](auto i_) {
                constexpr int i = CUBIC_CI(i_);
                const int n = P * i;
                v[i] = make_float2(__ldg(s0 + n), two ? __ldg(s1 + n) : 0.f);
            });
        }
    } else if constexpr (MODE == XM_INV) {
        static_for<0, E>([&](auto i_) {
            constexpr int i = CUBIC_CI(i_);
            a.dst[o0 + P * i] = v[i].x;
            if (two) a.dst[o1 + P * i] = v[i].y;
        });
    } else if constexpr (MODE == XM_RATIO) {
        const float eps = a.eps;
        const float *p0 = a.d + o0, *p1 = a.d + o1;
        if (a.nll_stats) {
            static_for<0, E>([&](auto i_) {
                constexpr int i = CUBIC_CI(i_);
                const int n = P * i;
                const float c0 = fmaxf(v[i].x, eps), c1 = fmaxf(v[i].y, eps);
                sum.nll = cf_add(sum.nll, c0 - __ldg(p0 + n) * logf(c0));
                if (two) sum.nll = cf_add(sum.nll, c1 - __ldg(p1 + n) * logf(c1));
            });
        }
        if (a.keep_a) {
            static_for<0, E>([&](auto i_) {
                constexpr int i = CUBIC_CI(i_);
                a.keep_a[o0 + P * i] = v[i].x;
                if (two) a.keep_a[o1 + P * i] = v[i].y;
            });
        }
        // fast division (max 2 ulp for denominators below 2^126; the clamp keeps them >= eps)
        static_for<0, E>([&](auto i_) {
            constexpr int i = CUBIC_CI(i_);
            const int n = P * i;
            const float x0 = __fdividef(__ldg(p0 + n), fmaxf(v[i].x, eps));
            const float x1 = __fdividef(two ? __ldg(p1 + n) : 0.f, fmaxf(v[i].y, eps));
            v[i] = make_float2(x0, x1);
        });
        if (center) {
            const float c = center->x;
            static_for<0, E>([&](auto i_) {
                constexpr int i = CUBIC_CI(i_);
                v[i] = make_float2(v[i].x - c, two ? v[i].y - c : 0.f);
            });
        }
        if (a.keep_b) {
            static_for<0, E>([&](auto i_) {
                constexpr int i = CUBIC_CI(i_);
                a.keep_b[o0 + P * i] = v[i].x;
                if (two) a.keep_b[o1 + P * i] = v[i].y;
            });
        }
    } else if constexpr (MODE == XM_UPDATE || MODE == XM_FINAL) {
        float *ob = (MODE == XM_FINAL || a.dst) ? a.dst : a.u;
        const float *p0 = a.u + o0, *p1 = a.u + o1;
        if (center) {
            const float h = center->y;
            static_for<0, E>([&](auto i_) { v[CUBIC_CI(i_)] = cadd(v[CUBIC_CI(i_)], make_float2(h, h)); });
        }
        if (a.keep_a) {
            static_for<0, E>([&](auto i_) {
                constexpr int i = CUBIC_CI(i_);
                a.keep_a[o0 + P * i] = v[i].x;
                if (two) a.keep_a[o1 + P * i] = v[i].y;
            });
        }
        const bool stats = a.stats != nullptr;
        const bool acc = MODE == XM_FINAL && a.acc_g != nullptr;
        if (acc) {
            // g = x - u in v's place until it is stored; the products with the previous g
            float2 u[E];
            static_for<0, E>([&](auto i_) {
                constexpr int i = CUBIC_CI(i_);
                u[i] = make_float2(p0[P * i], two ? p1[P * i] : 0.f);
            });
            static_for<0, E>([&](auto i_) {
                constexpr int i = CUBIC_CI(i_);
                const int n = P * i;
                const float h0 = a.acc_gprev ? __ldg(a.acc_gprev + o0 + n) : 0.f;
                const float h1 = a.acc_gprev && two ? __ldg(a.acc_gprev + o1 + n) : 0.f;
                const float x0 = u[i].x * v[i].x, x1 = u[i].y * v[i].y;
                const float g0 = x0 - u[i].x, g1 = x1 - u[i].y;
                if (a.acc_gprev) sum.acc_num = cf_add(cf_add(sum.acc_num, g0 * h0), g1 * h1);
                sum.acc_den = cf_add(cf_add(sum.acc_den, g0 * g0), g1 * g1);
                v[i] = make_float2(x0, x1);
                u[i] = make_float2(g0, g1);
            });
            static_for<0, E>([&](auto i_) {
                constexpr int i = CUBIC_CI(i_);
                const int n = P * i;
                a.acc_g[o0 + n] = u[i].x;
                if (two) a.acc_g[o1 + n] = u[i].y;
                ob[o0 + n] = v[i].x;
                if (two) ob[o1 + n] = v[i].y;
            });
        } else {
            // every load before the first store: u is usually updated in place
            static_for<0, E>([&](auto i_) {
                constexpr int i = CUBIC_CI(i_);
                const int n = P * i;
                const float u0 = p0[n], u1 = two ? p1[n] : 0.f;
                const float x0 = u0 * v[i].x, x1 = u1 * v[i].y;
                if (stats) {
                    sum.num = fmaf(x0 - u0, x0 - u0, fmaf(x1 - u1, x1 - u1, sum.num));
                    sum.den = fmaf(u0, u0, fmaf(u1, u1, sum.den));
                }
                v[i] = make_float2(x0, x1);
            });
            static_for<0, E>([&](auto i_) {
                constexpr int i = CUBIC_CI(i_);
                ob[o0 + P * i] = v[i].x;
                if (two) ob[o1 + P * i] = v[i].y;
            });
        }
    } else if constexpr (MODE == XM_ADJ_R) {
        // the formulas of x_body's XM_ADJ_R
        const float eps = a.eps;
        static_for<0, E>([&](auto i_) {
            constexpr int i = CUBIC_CI(i_);
            const int n = P * i;
            const float b0 = __ldg(a.adj_b + o0 + n), b1 = two ? __ldg(a.adj_b + o1 + n) : 0.f;
            const float d0 = __ldg(a.d + o0 + n), d1 = two ? __ldg(a.d + o1 + n) : 0.f;
            const float c0 = fmaxf(b0, eps), c1 = fmaxf(b1, eps);
            const float r0 = v[i].x, r1 = v[i].y;
            a.adj_dbar[o0 + n] += r0 / c0;
            if (two) a.adj_dbar[o1 + n] += r1 / c1;
            v[i] = make_float2(b0 > eps ? -r0 * d0 / (c0 * c0) : 0.f, b1 > eps ? -r1 * d1 / (c1 * c1) : 0.f);
        });
    } else if constexpr (MODE == XM_ADJ_U) {
        // the formulas of x_body's XM_ADJ_U
        if (a.adj_u) {
            static_for<0, E>([&](auto i_) {
                constexpr int i = CUBIC_CI(i_);
                const int n = P * i;
                const float x0 = v[i].x + a.adj_w[o0 + n], x1 = v[i].y + (two ? a.adj_w[o1 + n] : 0.f);
                v[i] = make_float2(x0 * __ldg(a.adj_u + o0 + n), x1 * (two ? __ldg(a.adj_u + o1 + n) : 0.f));
                a.adj_w[o0 + n] = x0 * __ldg(a.adj_q + o0 + n);
                if (two) a.adj_w[o1 + n] = x1 * __ldg(a.adj_q + o1 + n);
            });
        } else {
            static_for<0, E>([&](auto i_) {
                constexpr int i = CUBIC_CI(i_);
                a.adj_w[o0 + P * i] += v[i].x;
                if (two) a.adj_w[o1 + P * i] += v[i].y;
            });
        }
    }
}

// Adds the CTA's sums up: `unit` numbers the launch's CTAs; scratch: shared memory (16-byte
// aligned, 16 bytes a warp) that other threads may still be using.  Every thread calls it.
template <int MODE>
__device__ __forceinline__ void point_sums_finish(const XArgs &a, PointSums &sum, const int unit, float2 *scratch)
{
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int slot = (unit * (int)(blockDim.x >> 5) + warp) & 63;
    if constexpr (MODE == XM_RATIO) {
        if (a.nll_stats) {
            for (int o = 16; o > 0; o >>= 1)
                sum.nll = cf_merge(sum.nll, CFloat{__shfl_down_sync(0xffffffffu, sum.nll.s, o),
                                                   __shfl_down_sync(0xffffffffu, sum.nll.c, o)});
            if (lane == 0) {
                float *pair = a.nll_stats + 2 * slot;
                catomic_add(pair, pair + 1, sum.nll.s);
                catomic_add(pair, pair + 1, -sum.nll.c);
            }
        }
    }
    if constexpr (MODE == XM_UPDATE || MODE == XM_FINAL) {
        if (a.stats) {
            for (int o = 16; o > 0; o >>= 1) {
                sum.num += __shfl_down_sync(0xffffffffu, sum.num, o);
                sum.den += __shfl_down_sync(0xffffffffu, sum.den, o);
            }
            if (lane == 0) {
                float *st4 = a.stats + 4 * slot;
                catomic_add(st4, st4 + 1, sum.num);
                catomic_add(st4 + 2, st4 + 3, sum.den);
            }
        }
    }
    if constexpr (MODE == XM_FINAL) {
        if (a.acc_g) {  // uniform over the launch
            for (int o = 16; o > 0; o >>= 1) {
                sum.acc_num = cf_merge(sum.acc_num, CFloat{__shfl_down_sync(0xffffffffu, sum.acc_num.s, o),
                                                           __shfl_down_sync(0xffffffffu, sum.acc_num.c, o)});
                sum.acc_den = cf_merge(sum.acc_den, CFloat{__shfl_down_sync(0xffffffffu, sum.acc_den.s, o),
                                                           __shfl_down_sync(0xffffffffu, sum.acc_den.c, o)});
            }
            __syncthreads();  // the scratch is no longer in use
            float4 *red = reinterpret_cast<float4 *>(scratch);
            if (lane == 0) red[warp] = make_float4(sum.acc_num.s, sum.acc_num.c, sum.acc_den.s, sum.acc_den.c);
            __syncthreads();
            if (threadIdx.x == 0) {
                CFloat n{red[0].x, red[0].y}, d{red[0].z, red[0].w};
                for (int w = 1; w < (int)(blockDim.x >> 5); ++w) {
                    n = cf_merge(n, CFloat{red[w].x, red[w].y});
                    d = cf_merge(d, CFloat{red[w].z, red[w].w});
                }
                a.acc_part[unit] = make_float4(n.s, n.c, d.s, d.c);
            }
        }
    }
}

}  // namespace cubic
