// Fused form: the p-axis convolution kernel, and the plane kernels by mode.
#include "plane.cuh"

namespace cubic {

// mode ZM_CONV or ZM_CORR (a volume with a real H multiplies by it for both), or one of the
// one-way transforms.  72 registers: 28 warps per SM.
__global__ void __launch_bounds__(kConvWarps * 32, 7)
    k_conv(const __grid_constant__ ConvArgs one, const ConvTable *__restrict__ tab, int mode)
{
    extern __shared__ __align__(16) float2 smem_cv[];
    int b = blockIdx.x;
    const ConvArgs *ap = &one;
    if (tab) {
        const int v = find_volume(tab->prefix, tab->nvol, blockIdx.x);
        b -= (int)tab->prefix[v];
        ap = &tab->args[v];
    }
    const ConvArgs &a = *ap;
    // a volume with a real H multiplies by it for both convolution and correlation
    const int md = (a.Hr && (mode == ZM_CONV || mode == ZM_CORR)) ? (int)ZM_MUL_REAL : mode;
    len_switch(ConvLens{}, a.n, [&](auto n_) {
        constexpr int N = CUBIC_CI(n_);
        float2 *tw = smem_cv + conv_tile<N>() * kConvWarps;
        for (int i = threadIdx.x; i < Line<N>::kTw; i += blockDim.x) tw[i] = __ldg(a.tw + i);
        const int w = threadIdx.x >> 5;
        if (md <= ZM_CORR || md == ZM_MUL_REAL) {
            // a task's part of H is one piece: into L2 (a hint, before the wait)
            const int col0 = (b * kConvWarps + w) * conv_lines(N), left = a.mv - col0;
            if ((threadIdx.x & 31) == 0 && left > 0) {
                const unsigned n = (unsigned)((left < conv_lines(N) ? left : conv_lines(N)) * N) & ~3u;
                if (md == ZM_MUL_REAL)
                    bulk_prefetch_l2(a.Hr + col0 * N, n * 4u);
                else if (md != ZM_FWD_SCALE)
                    bulk_prefetch_l2(a.H + col0 * N, n * 8u);
            }
        }
        __syncthreads();
        pdl_wait();
        pdl_trigger();  // not before the wait: see k_plane
        conv_task<N>(a, md, b * kConvWarps + w, smem_cv + w * conv_tile<N>(), tw);
    });
}

cudaError_t launch_conv(const ConvArgs &a, const ConvTable *tab, int64_t blocks, int mode, size_t smem, cudaStream_t st)
{
    static cudaError_t attr = set_smem((const void *)k_conv, conv_smem(ConvLens{}));
    if (attr != cudaSuccess) return attr;
    if (blocks == 0) return cudaSuccess;
    return launch_pdl(k_conv, dim3((unsigned)blocks), dim3(kConvWarps * 32), smem, st, a, tab, mode);
}

cudaError_t launch_plane(int mode, const PlaneArgs &a, const PlaneTable *tab, int64_t blocks, int threads, size_t smem,
                         cudaStream_t st)
{
    switch (mode) {
    case XM_FWD: return launch_plane_mode<XM_FWD>(a, tab, blocks, threads, smem, st);
    case XM_INV: return launch_plane_mode<XM_INV>(a, tab, blocks, threads, smem, st);
    case XM_RATIO: return launch_plane_mode<XM_RATIO>(a, tab, blocks, threads, smem, st);
    case XM_UPDATE: return launch_plane_mode<XM_UPDATE>(a, tab, blocks, threads, smem, st);
    case XM_FINAL: return launch_plane_mode<XM_FINAL>(a, tab, blocks, threads, smem, st);
    case XM_ADJ_R: return launch_plane_mode<XM_ADJ_R>(a, tab, blocks, threads, smem, st);
    case XM_ADJ_U: return launch_plane_mode<XM_ADJ_U>(a, tab, blocks, threads, smem, st);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace cubic
