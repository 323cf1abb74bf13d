// The CTA-per-block FP32 kernel with two warps per block (fsr_coop.cuh), in a
// translation unit of its own to compile in parallel.
#include "fsr_coop.cuh"

namespace fsrk {
namespace {

template <int B>
cudaError_t configure_b() {
    const int bytes = (int)sizeof(coop::Smem<2>);
    const cudaFuncAttribute at = cudaFuncAttributeMaxDynamicSharedMemorySize;
    const cudaError_t e = cudaFuncSetAttribute(coop::fsr_coop_kernel<B, 2, true>, at, bytes);
    return e != cudaSuccess ? e : cudaFuncSetAttribute(coop::fsr_coop_kernel<B, 2, false>, at, bytes);
}

template <int B>
cudaError_t launch_b(const BatchArgs& a, const ImageArgs* one, cudaStream_t stream) {
    constexpr int T = coop::Cfg<2>::T;
    const size_t smem = sizeof(coop::Smem<2>);
    if (one) coop::fsr_coop_kernel<B, 2, true><<<(unsigned)a.total, T, smem, stream>>>(a, *one);
    else coop::fsr_coop_kernel<B, 2, false><<<(unsigned)a.total, T, smem, stream>>>(a, ImageArgs());
    return cudaGetLastError();
}

}  // namespace

cudaError_t configure_coop2() {
    cudaError_t e;
    if ((e = configure_b<2>()) != cudaSuccess) return e;
    if ((e = configure_b<4>()) != cudaSuccess) return e;
    if ((e = configure_b<8>()) != cudaSuccess) return e;
    return configure_b<16>();
}

cudaError_t launch_coop2(const BatchArgs& a, int B, const ImageArgs* one, cudaStream_t stream) {
    switch (B) {
        case 2: return launch_b<2>(a, one, stream);
        case 4: return launch_b<4>(a, one, stream);
        case 8: return launch_b<8>(a, one, stream);
        case 16: return launch_b<16>(a, one, stream);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace fsrk
