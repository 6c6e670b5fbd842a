// bp_launch_fp32.cu -- translation unit of the FP32 BP kernels.
#include "bp_launch.cuh"
namespace polar {
BPKernelInfo bp_kernel_info_fp32(int logn, int weighted, bool packed_syndrome)
{
    return bp_kernel_info_t<float>(logn, weighted, packed_syndrome);
}
BPKernelInfo bp_kernel_info_fp32_cyc(int logn, bool packed_syndrome)
{
    if (logn != 10) return {nullptr, 0, 0, 0};
    using KP = BPKernelPlan<10, 0, 4, 1>;
    using P = typename KP::Plan;
    constexpr int TH = KP::F * P::T;
    return {packed_syndrome ? (const void*)bp_kernel<10, float, 0, TH, true, 4> : (const void*)bp_kernel<10, float, 0, TH, false, 4>,
            TH, (size_t)KP::F * bp_slot_words<P, true>() * 4, KP::F};
}
cudaError_t wms_prepare_fp32(int logn, const float* w, int iters, void* out, cudaStream_t st)
{
    return wms_prepare_t<float>(logn, w, iters, out, st);
}
}  // namespace polar
