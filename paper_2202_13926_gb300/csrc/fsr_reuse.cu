// Re-use of reconstructed pixels (the sequential form of the original FSR
// that Sec. II leaves out): the wavefront kernel, FP32 and FP64, every B of
// the 32 x 32 support.  One warp per block of the wavefront (the launch
// shapes are in fsr_reuse.cuh), or for FP32 wavefronts of few blocks a CTA
// per block (fsr_coop.cuh): 16 1080p frames, K = 50: 103 -> 95 ms, 24: 120 ->
// 114 ms.  FP32 calls of few block rows take one launch for all wavefronts
// (fsr_coop_rows_kernel) unless they are captured: one 1080p frame, K = 100:
// 104.0 ms with a warp per block, 53.5 with a CTA per block and a launch per
// wavefront, 45.2 in one launch, 39.2 since its iteration is packed; six
// 480 x 270 frames 27.6, 14.7, 11.3 and 9.8 ms; all bit-identical.
#include "fsr_reuse.cuh"

namespace fsrk {

cudaError_t configure_reuse() {
    cudaError_t e;
    if ((e = configure_reuse_f32lo()) != cudaSuccess) return e;
    if ((e = configure_reuse_f32hi()) != cudaSuccess) return e;
    return configure_reuse_f64();
}

cudaError_t launch_reuse(const ReuseLaunch& a, int B, int fp64, int sm_count, cudaStream_t stream) {
    if (a.total <= 0) return cudaSuccess;
    if (fp64) return launch_reuse_f64(a, B, sm_count, stream);
    if (a.total <= (long long)kCoopReusePerSm * sm_count) return launch_coop_reuse(a, B, stream);
    if (B == 2 || B == 4) return launch_reuse_f32lo(a, B, sm_count, stream);
    return launch_reuse_f32hi(a, B, sm_count, stream);
}

}  // namespace fsrk
