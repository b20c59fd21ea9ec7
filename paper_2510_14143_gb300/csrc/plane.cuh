// plane.cuh -- the fused form of the passes for volumes whose planes fit on chip.
//
// A pass-by-pass convolution moves the spectrum through HBM six times (X, Y, Z, Y, X with
// the pointwise step in X).  Here one CTA keeps a whole plane -- all x, and all of a second
// axis c (z where possible, else y), at one index of the third axis p -- in shared memory
// and runs, in one kernel, the inverse c transform, the inverse x transform, the pointwise
// Richardson-Lucy step, the forward x transform and the forward c transform (k_plane).  A
// second kernel (k_conv) does the p axis: forward transform, product with H, inverse
// transform.  An iteration is then 4 launches instead of 8 and moves 52 bytes per voxel
// instead of 84 (a spectrum in and one out per kernel, H, and the pointwise operands), or 48
// instead of 80 with a real H.
//
// At these sizes a kernel visits its code once or twice, so instruction fetch (32 KB of
// first-level instruction cache) and latency bound it before anything else.  Hence:
//   - Every length is a product of two radices, N = R0 R1 (at most 16 each, but 125 = 5 x 25), and a
//     stage is a rolled loop over one radix butterfly per thread.  The loops' bodies are all
//     the code there is, and no thread holds more than one butterfly.
//   - Transforms are in place: decimation in frequency forward, decimation in time back, so
//     a line's frequencies stand in digit-reversed order (position k1 R1 + k2 holds
//     frequency k1 + R0 k2) and nothing is reordered.  Each thread rewrites the positions it
//     read, so an exchange needs one synchronisation instead of two; a convolution never
//     needs the natural order.
//   - The lines of a task belong to ONE warp: exchanges synchronise the warp, not the CTA.
//     A plane kernel has three CTA barriers: after its constants are copied, and between its c
//     and x parts (accelerated runs add two for their sums).
//   - Rows c and c + nc/2 share one complex line, z = row_c + i row_(c+nc/2).  Splitting
//     Z[k], Z[nx-k] into the two rows' spectra happens where the c transform loads them: the
//     thread that holds element c of frequency line k also holds element c + nc/2, so the
//     split is four additions and no exchange.  The plane needs nc/2 * nx complex slots,
//     the size of the real plane.  The halves of the split are left out; H carries the 1/2.
//   - k = 0 and k = nx/2 (real lines) ride as one complex line, line 0; its c transform is
//     separated into the two spectra on the way out.
//   - In HBM a plane's spectrum lies in the order the threads hold it (one register of
//     adjacent threads adjacent), so loads and stores are full-width whatever the lengths
//     are, with no row padding.  k_conv sees a matrix [np][M] of independent columns.  H has
//     the layout that k_conv's registers have between its two transforms.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>
#include <utility>

#include "line.cuh"
#include "registry.cuh"

namespace cubic {

// ------------------------------------------------------------------ length lists

template <int... Ns>
struct LenList {
    static constexpr bool has(int64_t len) { return ((len == Ns) || ...); }
};

// ------------------------------------------------------------------ plane geometry

// With h = ceil(nc/2) pair lines, line l of a plane's c transforms holds frequency k = l of
// the x axis: element c < h in slot k of pair line c, element c >= h in slot nx - k of pair
// line c - h.  Pair line m starts at m / R1 * bs + m % R1 * xs, R1 the c axis' second radix
// (bs = R1 xs for an odd nc).
struct PlaneGeo {
    int nx = 0, nc = 0, np = 0;   // x, in-plane second axis, planes (the p axis)
    int lines = 0;                // c lines: nx / 2 (even nx, line 0 carries k = 0 and nx / 2), or (nx + 1) / 2
    int xs = 0, bs = 0, cr1 = 0;  // pitch of a pair line, of cr1 = R1 pair lines (complex slots)
    // shared memory, in float2: [x twiddles][c twiddles][line slots][partners][center][plane];
    // what stands before the plane is copied from the plan's constant block, but for the center
    // (2 float2, one used)
    int off_twc = 0, off_tab = 0, off_neg = 0, off_plane = 0;
    int smem = 0;                 // bytes
    int mv = 0, m = 0;            // a plane's spectrum: values, and pitch (a multiple of 16)
    int rs = 0, ps = 0;           // real volume: elements between rows c and c + 1, between planes
};                                // (volumes of these lengths have fewer than 2^31 elements)

constexpr size_t kPlaneSmemMax = 227 * 1024;

struct PlaneArgs {
    XArgs x;            // operands of the pointwise step
    const float4 *tab;  // the constant block, g.off_plane float2
    PlaneGeo g;
};

// ------------------------------------------------------------------ c transforms of a plane

// Odd nc: rows c and c + h meet in no butterfly, so the split and the merge are passes of
// their own over the line's slots, in place (A in slot k, B in slot nx - k).
template <int NC, bool FWD>
__device__ __forceinline__ void plane_col_pairs(float2 *pk, float2 *pn, const int xs, const bool first, const bool evenx,
                                                const int m0, const int step)
{
    constexpr int h = (NC + 1) / 2;
#pragma unroll 1
    for (int m = m0; m < h; m += step) {
        float2 *zk = pk + m * xs, *zn = pn + m * xs;
        const float2 u = *zk, v = (FWD ? (first && !evenx) : m == h - 1) ? make_float2(0.f, 0.f) : *zn;
        if constexpr (FWD) {  // u = Z[k], v = Z[nx-k]
            const float s = evenx ? 1.f : 2.f;
            *zk = first ? make_float2(s * u.x, v.x) : make_float2(u.x + v.x, u.y - v.y);
            *zn = first ? make_float2(s * u.y, v.y) : make_float2(u.y + v.y, v.x - u.x);
        } else {  // the conjugates of A and B
            *zk = first ? make_float2(u.x, v.x) : make_float2(u.x + v.y, v.x - u.y);
            *zn = first ? make_float2(-u.y, -v.y) : make_float2(u.x - v.y, v.x + u.y);
        }
    }
}

// A task is Cw adjacent lines of one warp; butterfly i of a stage is line i % Cw, place i / Cw.
// A task's spectrum in HBM: register r of second-stage butterfly b of the line at c stands at
// r (cnt R0) + b cnt + c, cnt the task's lines.
template <int NC>
__device__ __forceinline__ void plane_col_inverse(const PlaneGeo &g, const float2 *__restrict__ spec, float2 *plane,
                                                  const float2 *twc, const uint32_t *tab)
{
    using F = Line<NC>;
    constexpr int R0 = F::R0, R1 = F::R1, H = R0 / 2, Cw = col_lines(NC);
    const int lane = threadIdx.x & 31, W = blockDim.x >> 5, xs = g.xs, bs = g.bs;
    const int c = lane % Cw;
    const bool evenx = (g.nx & 1) == 0;
    // where element (or position) pos of a line stands, for an odd nc
    auto at = [&](float2 *k, float2 *n, int pos) {
        constexpr int h = (NC + 1) / 2;
        return pos < h ? k + pos * xs : n + (pos - h) * xs;
    };
    for (int l0 = (threadIdx.x >> 5) * Cw; l0 < g.lines; l0 += W * Cw) {
        const int cnt = min(Cw, g.lines - l0);
        const bool ok = c < cnt, first = l0 + c == 0;
        const uint32_t sl = ok ? tab[l0 + c] : 0u;
        float2 *pk = plane + (sl & 0xffffu), *pn = plane + (sl >> 16);
        const float2 *src = spec + l0 * NC;
        if (ok) {
#pragma unroll 1
            for (int b = lane / Cw; b < R0; b += 32 / Cw) {
                float2 x[R1];
                static_for<0, R1>([&](auto r_) { x[CUBIC_CI(r_)] = cconj(src[CUBIC_CI(r_) * (cnt * R0) + b * cnt + c]); });
                if (first && evenx) {
                    // line 0 carries both real lines: V = D + i N (here conjugated)
                    const float2 *ny = spec + g.lines * NC + b;
                    static_for<0, R1>([&](auto r_) {
                        const float2 f = ny[CUBIC_CI(r_) * R0];
                        x[CUBIC_CI(r_)] = make_float2(x[CUBIC_CI(r_)].x - f.y, x[CUBIC_CI(r_)].y - f.x);
                    });
                }
                Dft<R1, kPacked>::run(x);
                if constexpr (NC % 2) {
                    static_for<0, R1>([&](auto r_) { *at(pk, pn, b * R1 + CUBIC_CI(r_)) = x[CUBIC_CI(r_)]; });
                } else {
                    float2 *q = b < H ? pk + b * bs : pn + (b - H) * bs;
                    static_for<0, R1>([&](auto r_) { q[CUBIC_CI(r_) * xs] = x[CUBIC_CI(r_)]; });
                }
            }
        }
        __syncwarp();
        if (NC % 2) {
            if (ok) {
#pragma unroll 1
                for (int j = lane / Cw; j < R1; j += 32 / Cw) {
                    float2 x[R0];
                    static_for<0, R0>([&](auto r_) { x[CUBIC_CI(r_)] = *at(pk, pn, j + CUBIC_CI(r_) * R1); });
                    F::bwd0(x, twc, j);
                    static_for<0, R0>([&](auto r_) { *at(pk, pn, j + CUBIC_CI(r_) * R1) = x[CUBIC_CI(r_)]; });
                }
            }
            __syncwarp();
            if (ok) plane_col_pairs<NC, false>(pk, pn, xs, first, evenx, lane / Cw, 32 / Cw);
        } else if (ok) {
#pragma unroll 1
            for (int j = lane / Cw; j < R1; j += 32 / Cw) {
                float2 x[R0];
                float2 *k0 = pk + j * xs, *n0 = pn + j * xs;
                static_for<0, H>([&](auto r_) {
                    x[CUBIC_CI(r_)] = k0[CUBIC_CI(r_) * bs];
                    x[CUBIC_CI(r_) + H] = n0[CUBIC_CI(r_) * bs];
                });
                F::bwd0(x, twc, j);
                // x is the conjugate of the line; rows A = x[r], B = x[r + H] merge into
                // Z[k] = A + iB and Z[nx-k] = conj A + i conj B
                if (first) {
                    static_for<0, H>([&](auto r_) {
                        constexpr int r = CUBIC_CI(r_);
                        k0[r * bs] = make_float2(x[r].x, x[r + H].x);
                        n0[r * bs] = make_float2(-x[r].y, -x[r + H].y);
                    });
                } else {
                    static_for<0, H>([&](auto r_) {
                        constexpr int r = CUBIC_CI(r_);
                        const float2 u = x[r], v = x[r + H];
                        k0[r * bs] = make_float2(u.x + v.y, v.x - u.y);
                        n0[r * bs] = make_float2(u.x - v.y, v.x + u.y);
                    });
                }
            }
        }
    }
}

template <int NC>
__device__ __forceinline__ void plane_col_forward(const PlaneGeo &g, float2 *__restrict__ spec, float2 *plane,
                                                  const float2 *twc, const uint32_t *tab, const uint32_t *neg)
{
    using F = Line<NC>;
    constexpr int R0 = F::R0, R1 = F::R1, H = R0 / 2, Cw = col_lines(NC);
    const int lane = threadIdx.x & 31, W = blockDim.x >> 5, xs = g.xs, bs = g.bs;
    const int c = lane % Cw;
    const bool evenx = (g.nx & 1) == 0;
    // where element (or position) pos of a line stands, for an odd nc
    auto at = [&](float2 *k, float2 *n, int pos) {
        constexpr int h = (NC + 1) / 2;
        return pos < h ? k + pos * xs : n + (pos - h) * xs;
    };
    for (int l0 = (threadIdx.x >> 5) * Cw; l0 < g.lines; l0 += W * Cw) {
        const int cnt = min(Cw, g.lines - l0);
        const bool ok = c < cnt, first = l0 + c == 0;
        const uint32_t sl = ok ? tab[l0 + c] : 0u;
        float2 *pk = plane + (sl & 0xffffu), *pn = plane + (sl >> 16);
        float2 *dst = spec + l0 * NC;
        if (NC % 2) {
            if (ok) plane_col_pairs<NC, true>(pk, pn, xs, first, evenx, lane / Cw, 32 / Cw);
            __syncwarp();
            if (ok) {
#pragma unroll 1
                for (int j = lane / Cw; j < R1; j += 32 / Cw) {
                    float2 x[R0];
                    static_for<0, R0>([&](auto r_) { x[CUBIC_CI(r_)] = *at(pk, pn, j + CUBIC_CI(r_) * R1); });
                    F::fwd0(x, twc, j);
                    static_for<0, R0>([&](auto r_) { *at(pk, pn, j + CUBIC_CI(r_) * R1) = x[CUBIC_CI(r_)]; });
                }
            }
        } else if (ok) {
#pragma unroll 1
            for (int j = lane / Cw; j < R1; j += 32 / Cw) {
                float2 x[R0];
                float2 *k0 = pk + j * xs, *n0 = pn + j * xs;
                // 2 A and 2 B; line 0: D + i N unscaled (the separation below doubles it), or
                // 2 D where nx is odd
                if (first) {
                    const float s = evenx ? 1.f : 2.f, e = evenx ? 1.f : 0.f;
                    static_for<0, H>([&](auto r_) {
                        constexpr int r = CUBIC_CI(r_);
                        const float2 z = k0[r * bs], n = evenx ? n0[r * bs] : make_float2(0.f, 0.f);
                        x[r] = make_float2(s * z.x, e * n.x);
                        x[r + H] = make_float2(s * z.y, e * n.y);
                    });
                } else {
                    static_for<0, H>([&](auto r_) {
                        constexpr int r = CUBIC_CI(r_);
                        const float2 z = k0[r * bs], n = n0[r * bs];
                        x[r] = make_float2(z.x + n.x, z.y - n.y);
                        x[r + H] = make_float2(z.y + n.y, n.x - z.x);
                    });
                }
                F::fwd0(x, twc, j);
                static_for<0, H>([&](auto r_) {
                    k0[CUBIC_CI(r_) * bs] = x[CUBIC_CI(r_)];
                    n0[CUBIC_CI(r_) * bs] = x[CUBIC_CI(r_) + H];
                });
            }
        }
        __syncwarp();
        if (ok) {
#pragma unroll 1
            for (int b = lane / Cw; b < R0; b += 32 / Cw) {
                float2 x[R1];
                auto q = [&](int r) {
                    if constexpr (NC % 2) return at(pk, pn, b * R1 + r);
                    return (b < H ? pk + b * bs : pn + (b - H) * bs) + r * xs;
                };
                static_for<0, R1>([&](auto r_) { x[CUBIC_CI(r_)] = *q(CUBIC_CI(r_)); });
                Dft<R1, kPacked>::run(x);
                if (first && evenx) {
                    static_for<0, R1>([&](auto r_) { *q(CUBIC_CI(r_)) = x[CUBIC_CI(r_)]; });
                } else {
                    static_for<0, R1>([&](auto r_) { dst[CUBIC_CI(r_) * (cnt * R0) + b * cnt + c] = x[CUBIC_CI(r_)]; });
                }
            }
        }
        if (l0 == 0 && evenx) {
            // line 0: D(q) = V(q) + conj V(-q), N(q) = (V(q) - conj V(-q)) / i, both doubled;
            // neg: where V(-q) stands, relative to slot k (top bit: to slot nx - k)
            const uint32_t s0 = tab[0];
            float2 *z0 = plane + (s0 & 0xffffu), *z1 = plane + (s0 >> 16);
            float2 *ny = spec + g.lines * NC;
            __syncwarp();
#pragma unroll 1
            for (int pos = lane; pos < NC; pos += 32) {
                const int b = pos / R1, r = pos % R1;
                const float2 v = NC % 2 ? *at(z0, z1, pos) : (b < H ? z0 + b * bs : z1 + (b - H) * bs)[r * xs];
                const uint32_t o = neg[pos];
                const float2 m = ((o >> 31) ? z1 : z0)[o & 0x7fffffffu];
                dst[r * (cnt * R0) + b * cnt] = make_float2(v.x + m.x, v.y - m.y);
                ny[r * R0 + b] = make_float2(v.y + m.y, m.x - v.x);
            }
        }
    }
}

// ------------------------------------------------------------------ x transforms of a plane

// x lines of the plane.  A task is Lw pair lines of one warp; butterfly i of a stage is place
// i % (butterflies per line) of line i / that.  spec: the plane's spectrum is in shared
// memory (false: the step starts from zeros, XM_ADJ_U); back: transform the result.
template <int NX, int MODE>
__device__ __forceinline__ void plane_rows(const PlaneArgs &a, float2 *plane, const float2 *twx, const int p,
                                           const bool spec, const bool back, PointSums &sum, const float2 *center)
{
    using F = Line<NX>;
    constexpr int R0 = F::R0, R1 = F::R1, Lw = row_lines(NX);
    const int lane = threadIdx.x & 31, W = blockDim.x >> 5;
    const int H = (a.g.nc + 1) / 2, xs = a.g.xs, bs = a.g.bs, cr1 = a.g.cr1;
    const int rs = a.g.rs, second = H * rs, off = p * a.g.ps;
    for (int m0 = (threadIdx.x >> 5) * Lw; m0 < H; m0 += W * Lw) {
        const int cnt = min(Lw, H - m0);
        auto line = [&](int l) {
            const int m = m0 + l, q = m / cr1;
            return plane + q * bs + (m - q * cr1) * xs;
        };
        if (MODE != XM_FWD && spec) {
#pragma unroll 1
            for (int i = lane; i < cnt * R0; i += 32) {
                float2 *q = line(i / R0) + i % R0 * F::kStep;
                float2 x[R1];
                static_for<0, R1>([&](auto r_) { x[CUBIC_CI(r_)] = cconj(q[CUBIC_CI(r_)]); });
                Dft<R1, kPacked>::run(x);
                static_for<0, R1>([&](auto r_) { q[CUBIC_CI(r_)] = x[CUBIC_CI(r_)]; });
            }
            __syncwarp();
        }
#pragma unroll 1
        for (int i = lane; i < cnt * R1; i += 32) {
            const int l = i / R1, j = i % R1;
            float2 *q = line(l) + j;
            float2 x[R0];
            if (MODE != XM_FWD) {
                if (spec) {
                    static_for<0, R0>([&](auto r_) { x[CUBIC_CI(r_)] = q[CUBIC_CI(r_) * F::kStep]; });
                    F::bwd0(x, twx, j);
                    static_for<0, R0>([&](auto r_) { x[CUBIC_CI(r_)].y = -x[CUBIC_CI(r_)].y; });
                } else {
                    static_for<0, R0>([&](auto r_) { x[CUBIC_CI(r_)] = make_float2(0.f, 0.f); });
                }
            }
            const int o = off + (m0 + l) * rs + j;
            // the last line of an odd nc has one row
            plane_point<MODE, R0, R1>(a.x, x, o, o + second, m0 + l + H < a.g.nc, sum, center);
            if (MODE != XM_INV && MODE != XM_FINAL && back) {
                F::fwd0(x, twx, j);
                static_for<0, R0>([&](auto r_) { q[CUBIC_CI(r_) * F::kStep] = x[CUBIC_CI(r_)]; });
            }
        }
        if (MODE != XM_INV && MODE != XM_FINAL && back) {
            __syncwarp();
#pragma unroll 1
            for (int i = lane; i < cnt * R0; i += 32) {
                float2 *q = line(i / R0) + i % R0 * F::kStep;
                float2 x[R1];
                static_for<0, R1>([&](auto r_) { x[CUBIC_CI(r_)] = q[CUBIC_CI(r_)]; });
                Dft<R1, kPacked>::run(x);
                static_for<0, R1>([&](auto r_) { q[CUBIC_CI(r_)] = x[CUBIC_CI(r_)]; });
            }
        }
    }
}

// ------------------------------------------------------------------ the lengths

using PlaneX = LenList<32, 36, 40, 45, 48, 50, 54, 60, 64, 72, 75, 80, 81, 90, 96, 100, 108, 120, 125, 128, 135, 144, 150,
                       160, 192>;
using PlaneC = LenList<8, 10, 12, 16, 18, 20, 24, 30, 32, 36, 40, 45, 48, 50, 54, 60, 64, 72, 75, 80, 81, 90, 96, 100,
                       108, 120, 125, 128, 135, 144, 150, 160, 192>;
using ConvLens = LenList<8, 9, 10, 12, 15, 16, 18, 20, 24, 25, 27, 30, 32, 36, 40, 45, 48, 50, 54, 60, 64, 72, 75, 80, 81,
                         90, 96, 100, 108, 120, 125, 128, 135, 144, 150, 160, 192>;

// The plane kernels are held to 80 registers: 24 warps per SM
constexpr int kPlaneThreads = 768;

// calls f(std::integral_constant<int, N>{}) for the N of the (ascending) list equal to n, by
// bisection: a kernel dispatches two or three times, and a comparison costs as much as an
// instruction that works
template <int... Ns>
struct LenArray {
    static constexpr int n = sizeof...(Ns);
    static constexpr int v[n] = {Ns...};
};
template <class A, int Lo, int Hi, class F>
__device__ __forceinline__ void bisect(int n, F &&f)
{
    if constexpr (Hi - Lo == 1) {
        constexpr int len = A::v[Lo];
        if (n == len) f(std::integral_constant<int, len>{});
    } else {
        constexpr int Mid = (Lo + Hi) / 2, len = A::v[Mid];
        if (n < len)
            bisect<A, Lo, Mid>(n, f);
        else
            bisect<A, Mid, Hi>(n, f);
    }
}
template <int... Ns, class F>
__device__ __forceinline__ void len_switch(LenList<Ns...>, int n, F &&f)
{
    bisect<LenArray<Ns...>, 0, (int)sizeof...(Ns)>(n, f);
}

// runtime copies of the per-length constants (r1 = 0: the list lacks the length)
struct PlaneLen {
    int r0 = 0, r1 = 0, slots = 0, tw = 0, row_lines = 0, col_lines = 0, conv_lines = 0;
};
template <int... Ns>
inline PlaneLen plane_len(LenList<Ns...>, int64_t n)
{
    PlaneLen r;
    (void)((n == Ns ? (r = PlaneLen{Line<Ns>::R0, Line<Ns>::R1, Line<Ns>::kSlots, Line<Ns>::kTw, row_lines(Ns), col_lines(Ns),
                                     conv_lines(Ns)},
                       true)
                    : false) ||
           ...);
    return r;
}

// Planes of several volumes in one launch: volume v's planes are blocks
// prefix[v] .. prefix[v + 1) - 1.
struct PlaneTable {
    int nvol;
    int64_t prefix[kMaxBatch + 1];
    PlaneArgs args[kMaxBatch];
};

// ------------------------------------------------------------------ constant blocks

// A plan's constants, written once: the plane kernel's block (see PlaneGeo) and, after it,
// the stage twiddles of the p axis.  wx, wc, wp: the axes' tables W_N^m.  One CTA.
__device__ __forceinline__ void plane_tables(const PlaneGeo &g, float2 *tab, const float2 *wx, const float2 *wc,
                                             const float2 *wp)
{
    uint32_t *slots = reinterpret_cast<uint32_t *>(tab + g.off_tab), *neg = reinterpret_cast<uint32_t *>(tab + g.off_neg);
    len_switch(PlaneX{}, g.nx, [&](auto n_) {
        constexpr int N = CUBIC_CI(n_);
        using F = Line<N>;
        F::fill_twiddles(tab, wx, threadIdx.x, blockDim.x);
        for (int l = threadIdx.x; l < g.lines; l += blockDim.x) {
            // slots of frequency l and of its partner: nx - l; for line 0 nx / 2 (even nx), or
            // the spare slot past the line
            const int k = F::slot(F::pos_of(l));
            const int n = l > 0 ? F::slot(F::pos_of(N - l)) : N % 2 == 0 ? F::slot(F::pos_of(N / 2)) : F::kSlots;
            slots[l] = (uint32_t)k | (uint32_t)n << 16;
        }
    });
    len_switch(PlaneC{}, g.nc, [&](auto n_) {
        constexpr int N = CUBIC_CI(n_);
        using F = Line<N>;
        F::fill_twiddles(tab + g.off_twc, wc, threadIdx.x, blockDim.x);
        for (int pos = threadIdx.x; pos < N; pos += blockDim.x) {
            // where the value at minus this position's frequency stands in its line
            const int f = F::freq_of(pos), q = F::pos_of(f == 0 ? 0 : N - f);
            const int h = (N + 1) / 2, half = q >= h, m = q - half * h;
            neg[pos] = (uint32_t)(m / F::R1 * g.bs + m % F::R1 * g.xs) | (uint32_t)half << 31;
        }
    });
    len_switch(ConvLens{}, g.np,
                  [&](auto n_) { Line<CUBIC_CI(n_)>::fill_twiddles(tab + g.off_plane, wp, threadIdx.x, blockDim.x); });
}

// ------------------------------------------------------------------ kernels

// 8 bytes from global to shared memory, asynchronously; and the wait for this thread's copies
__device__ __forceinline__ void copy_async8(void *dst, const void *src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}
__device__ __forceinline__ void copy_async_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

template <int MODE>
__global__ void __launch_bounds__(kPlaneThreads, 1)
    k_plane(const __grid_constant__ PlaneArgs one, const PlaneTable *__restrict__ tab)
{
    extern __shared__ __align__(16) float2 smem_pl[];
    int p = blockIdx.x;
    const PlaneArgs *ap = &one;
    if (tab) {
        const int v = find_volume(tab->prefix, tab->nvol, blockIdx.x);
        p -= (int)tab->prefix[v];
        ap = &tab->args[v];
    }
    const PlaneArgs &a = *ap;
    const PlaneGeo g = a.g;
    const float2 *twx = smem_pl, *twc = smem_pl + g.off_twc;
    const uint32_t *slots = reinterpret_cast<const uint32_t *>(smem_pl + g.off_tab);
    const uint32_t *neg = reinterpret_cast<const uint32_t *>(smem_pl + g.off_neg);
    float2 *plane = smem_pl + g.off_plane;
    constexpr bool kIn = MODE != XM_FWD, kOut = MODE != XM_INV && MODE != XM_FINAL;
    constexpr bool kCenter = MODE == XM_RATIO || MODE == XM_UPDATE || MODE == XM_FINAL;
    float2 *center = kCenter && a.x.center ? plane - 2 : nullptr;

    // constants of the plan: before the wait
    for (int i = threadIdx.x; i < g.off_plane / 2; i += blockDim.x)
        reinterpret_cast<float4 *>(smem_pl)[i] = __ldg(a.tab + i);
    if constexpr (MODE == XM_RATIO || MODE == XM_UPDATE || MODE == XM_FINAL) {
        // bring the operand rows into L2 while the spectrum is on its way (a hint, so before
        // the wait; nothing in the plane's way needs them for a few microseconds)
        if (g.nx % 4 == 0) {
            const float *op = (MODE == XM_RATIO ? a.x.d : a.x.u) + p * g.ps;
            for (int r = threadIdx.x; r < g.nc; r += blockDim.x) bulk_prefetch_l2(op + r * g.rs, (unsigned)g.nx * 4u);
        }
    }
    __syncthreads();
    pdl_wait();
    // the center on its way under the loads of the spectrum, in shared memory and not in a register:
    // loaded where it is used it cost 0.5 us a launch
    if (kCenter && center && threadIdx.x == 0) copy_async8(center, a.x.center);

    const bool spec = kIn && (MODE != XM_ADJ_U || a.x.spec_in != nullptr);
    const bool back = kOut && (MODE != XM_ADJ_U || a.x.adj_u != nullptr);
    if constexpr (kIn) {
        if (spec) {
            len_switch(PlaneC{}, g.nc,
                       [&](auto n_) { plane_col_inverse<CUBIC_CI(n_)>(g, a.x.spec_in + p * g.m, plane, twc, slots); });
            if (kCenter) copy_async_wait();
            __syncthreads();
        }
    }
    // The next kernel's CTAs may come now.  Released at the start, they would take their places
    // while this kernel's predecessor still drains, several on the SMs that empty first
    // (128x64x128 voxels, 256 threads: 43.9 us an iteration, 28.2 us with the release here).
    pdl_trigger();
    PointSums sum;
    len_switch(PlaneX{}, g.nx, [&](auto n_) { plane_rows<CUBIC_CI(n_), MODE>(a, plane, twx, p, spec, back, sum, center); });
    if constexpr (kOut) {
        if (back) {
            __syncthreads();
            len_switch(PlaneC{}, g.nc,
                          [&](auto n_) { plane_col_forward<CUBIC_CI(n_)>(g, a.x.spec_out + p * g.m, plane, twc, slots, neg); });
        }
    }
    point_sums_finish<MODE>(a.x, sum, p, plane);
}

// ------------------------------------------------------------------ p axis: convolution

struct ConvArgs {
    float2 *spec;        // [n][m], columns 0 .. mv - 1 valid
    const float2 *H;     // native order of the transformed lines (see conv_index)
    const float *Hr;     // the same for a real H (ZM_MUL_REAL)
    const float2 *tw;    // stage twiddles
    int m, mv;
    int n;
    float scale;         // ZM_FWD_SCALE (natural in, native out) and ZM_INV_SCALE (the reverse)
    // the reverse sweep's extras, as in ZArgs, in native order
    float2 *save, *gacc;
    const float2 *gother;
    int gconj;
    float2 *out;         // ZM_FWD_SCALE: the native-order result; ZM_INV_SCALE: its input
};

struct ConvTable {
    int nvol;
    int64_t prefix[kMaxBatch + 1];
    ConvArgs args[kMaxBatch];
};

constexpr int kConvWarps = 4;

// One warp transforms Cw adjacent columns, loading straight into registers and exchanging
// through its own tile of shared memory (position p of column c at slot(p) Cw + c), so
// nothing waits at a CTA barrier.  The second forward stage, the product and the first
// inverse stage are one loop.
template <int N>
__device__ __forceinline__ void conv_task(const ConvArgs &a, const int mode, const int task, float2 *sm, const float2 *tw)
{
    using F = Line<N>;
    constexpr int R0 = F::R0, R1 = F::R1, Cw = conv_lines(N);
    const int lane = threadIdx.x & 31, c = lane % Cw;
    const int col0 = task * Cw, m = a.m;
    if (col0 >= a.mv) return;  // uniform over the warp
    const int cnt = min(Cw, a.mv - col0);
    const bool ok = c < cnt;
    float2 *col = a.spec + col0 + c, *tile = sm + c;
    const int nat = col0 * N + c;  // native order: register r of butterfly b at r (cnt R0) + b cnt
    if (mode != ZM_INV_SCALE && ok) {
#pragma unroll 1
        for (int j = lane / Cw; j < R1; j += 32 / Cw) {
            float2 x[R0];
            static_for<0, R0>([&](auto r_) { x[CUBIC_CI(r_)] = col[(j + CUBIC_CI(r_) * R1) * m]; });
            F::fwd0(x, tw, j);
            static_for<0, R0>([&](auto r_) { tile[(j + CUBIC_CI(r_) * F::kStep) * Cw] = x[CUBIC_CI(r_)]; });
        }
    }
    __syncwarp();
    if (ok) {
#pragma unroll 1
        for (int b = lane / Cw; b < R0; b += 32 / Cw) {
            float2 *q = tile + b * F::kStep * Cw;
            const int at = nat + b * cnt;
            const int step = cnt * R0;
            float2 x[R1];
            if (mode == ZM_INV_SCALE) {
                static_for<0, R1>([&](auto r_) { x[CUBIC_CI(r_)] = cconj(a.out[at + CUBIC_CI(r_) * step]); });
            } else {
                static_for<0, R1>([&](auto r_) { x[CUBIC_CI(r_)] = q[CUBIC_CI(r_) * Cw]; });
                Dft<R1, kPacked>::run(x);
                if (mode == ZM_FWD_SCALE) {
                    static_for<0, R1>([&](auto r_) { a.out[at + CUBIC_CI(r_) * step] = cscale(x[CUBIC_CI(r_)], a.scale); });
                    continue;
                }
                if (a.save) static_for<0, R1>([&](auto r_) { a.save[at + CUBIC_CI(r_) * step] = x[CUBIC_CI(r_)]; });
                if (a.gacc) {
                    static_for<0, R1>([&](auto r_) {
                        const int i = at + CUBIC_CI(r_) * step;
                        const float2 o = __ldg(a.gother + i), v = x[CUBIC_CI(r_)];
                        a.gacc[i] = cadd(a.gacc[i], a.gconj ? cmulconj(o, v) : cmulconj(v, o));
                    });
                }
                // product with H or conj(H), then conjugate for the inverse transform
                if (mode == ZM_MUL_REAL) {
                    static_for<0, R1>([&](auto r_) {
                        const float h = __ldg(a.Hr + at + CUBIC_CI(r_) * step);
                        x[CUBIC_CI(r_)] = make_float2(x[CUBIC_CI(r_)].x * h, -x[CUBIC_CI(r_)].y * h);
                    });
                } else {
                    const float s = mode == ZM_CORR ? -1.f : 1.f;
                    static_for<0, R1>([&](auto r_) {
                        float2 h = __ldg(a.H + at + CUBIC_CI(r_) * step);
                        h.y *= s;
                        x[CUBIC_CI(r_)] = cconj(cmul(x[CUBIC_CI(r_)], h));
                    });
                }
            }
            Dft<R1, kPacked>::run(x);
            static_for<0, R1>([&](auto r_) { q[CUBIC_CI(r_) * Cw] = x[CUBIC_CI(r_)]; });
        }
    }
    if (mode == ZM_FWD_SCALE) return;
    __syncwarp();
    if (ok) {
        const float sx = mode == ZM_INV_SCALE ? a.scale : 1.f;
#pragma unroll 1
        for (int j = lane / Cw; j < R1; j += 32 / Cw) {
            float2 x[R0];
            static_for<0, R0>([&](auto r_) { x[CUBIC_CI(r_)] = tile[(j + CUBIC_CI(r_) * F::kStep) * Cw]; });
            F::bwd0(x, tw, j);
            static_for<0, R0>([&](auto r_) {
                col[(j + CUBIC_CI(r_) * R1) * m] = make_float2(x[CUBIC_CI(r_)].x * sx, -x[CUBIC_CI(r_)].y * sx);
            });
        }
    }
}

// shared memory of one warp's tile, and of a CTA with its twiddles, in float2
template <int N>
constexpr int conv_tile() { return Line<N>::kSlots * conv_lines(N); }
template <int N>
constexpr int conv_smem_one() { return conv_tile<N>() * kConvWarps + Line<N>::kTw; }

template <int... Ns>
constexpr size_t conv_smem(LenList<Ns...>)
{
    size_t m = 0;
    ((m = conv_smem_one<Ns>() * sizeof(float2) > m ? conv_smem_one<Ns>() * sizeof(float2) : m), ...);
    return m;
}
template <int... Ns>
inline size_t conv_smem_of(LenList<Ns...>, int64_t n)
{
    size_t r = 0;
    (void)((n == Ns ? (r = conv_smem_one<Ns>() * sizeof(float2), true) : false) || ...);
    return r;
}
inline int64_t conv_blocks_of(const PlaneLen &l, int64_t mv)
{
    const int64_t cols = (int64_t)l.conv_lines * kConvWarps;
    return (mv + cols - 1) / cols;
}

// ------------------------------------------------------------------ launchers

// One translation unit per mode (plane_*.cu).  tab == nullptr: the planes of `a`.
template <int MODE>
cudaError_t launch_plane_mode(const PlaneArgs &a, const PlaneTable *tab, int64_t blocks, int threads, size_t smem,
                              cudaStream_t st);

#define CUBIC_PLANE_UNIT(MODE)                                                                                 \
    template <>                                                                                                \
    cudaError_t launch_plane_mode<MODE>(const PlaneArgs &a, const PlaneTable *tab, int64_t blocks, int threads, \
                                        size_t smem, cudaStream_t st)                                          \
    {                                                                                                          \
        static cudaError_t attr = set_smem((const void *)k_plane<MODE>, kPlaneSmemMax);                        \
        if (attr != cudaSuccess) return attr;                                                                  \
        if (blocks == 0) return cudaSuccess;                                                                   \
        return launch_pdl(k_plane<MODE>, dim3((unsigned)blocks), dim3(threads), smem, st, a, tab);             \
    }

cudaError_t launch_plane(int mode, const PlaneArgs &a, const PlaneTable *tab, int64_t blocks, int threads, size_t smem,
                         cudaStream_t st);
cudaError_t launch_conv(const ConvArgs &a, const ConvTable *tab, int64_t blocks, int mode, size_t smem, cudaStream_t st);

}  // namespace cubic
