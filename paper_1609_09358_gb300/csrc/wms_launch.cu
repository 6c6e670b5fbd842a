// wms_launch.cu -- translation unit of the training kernels (see wms_kernels.cuh).
#define POLAR_WMS_KERNELS
#include "wms_kernels.cuh"

namespace polar {

// CF, CB: resident CTAs per SM the forward and the backward kernel are allocated for.
template <int LOGN, int CF, int CB>
static cudaError_t wms_launch_t(bool backward, const WMSArgs& a, cudaStream_t st)
{
    using P = typename BPConfig<LOGN>::Plan;
    constexpr int F = wms_frames_per_cta<P>(), TH = F * P::T;
    static_assert(plan_is_conflict_free<P>(), "exchange layout has bank conflicts");
    static_assert(P::xidx_l(0) % 2 == 0, "odd number of exchanges per iteration");
    const unsigned grid = (unsigned)((a.B + F - 1) / F);
    const size_t words = (size_t)F * (backward ? wms_slot_floats<P>() : 2 * P::XW);
    const size_t smem = words * sizeof(float);
    static_assert((size_t)F * wms_slot_floats<P>() * sizeof(float) <= 48 * 1024 || LOGN == 11, "default limit");
    if (backward) {
        const cudaError_t e = raise_smem_limit((const void*)wms_backward_kernel<P, TH, CB>, smem);
        if (e != cudaSuccess) return e;
        wms_backward_kernel<P, TH, CB><<<grid, TH, smem, st>>>(a);
    } else {
        wms_forward_kernel<P, TH, CF><<<grid, TH, smem, st>>>(a);
    }
    return cudaGetLastError();
}

static cudaError_t wms_launch(int logn, bool backward, const WMSArgs& a, cudaStream_t st)
{
    switch (logn) {
        case 7: return wms_launch_t<7, 4, 4>(backward, a, st);
        case 8: return wms_launch_t<8, 3, 3>(backward, a, st);
        case 9: return wms_launch_t<9, 6, 6>(backward, a, st);
        case 10: return wms_launch_t<10, 3, 3>(backward, a, st);
        default: return wms_launch_t<11, 1, 1>(backward, a, st);
    }
}

cudaError_t wms_forward_launch(int logn, const WMSArgs& a, cudaStream_t st) { return wms_launch(logn, false, a, st); }
cudaError_t wms_backward_launch(int logn, const WMSArgs& a, cudaStream_t st) { return wms_launch(logn, true, a, st); }

}  // namespace polar
