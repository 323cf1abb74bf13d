// Instantiations and launches of the CTA-per-block FP32 kernels (fsr_coop.cuh).
#include <algorithm>

#include "fsr_coop.cuh"

namespace fsrk {
namespace {

template <int B>
cudaError_t configure_b() {
    cudaError_t e;
    const int bytes = (int)sizeof(coop::Smem<4>);
    const cudaFuncAttribute at = cudaFuncAttributeMaxDynamicSharedMemorySize;
    if ((e = cudaFuncSetAttribute(coop::fsr_coop_kernel<B, 4, true>, at, bytes)) != cudaSuccess) return e;
    if ((e = cudaFuncSetAttribute(coop::fsr_coop_kernel<B, 4, false>, at, bytes)) != cudaSuccess) return e;
    if ((e = cudaFuncSetAttribute(coop::fsr_coop_reuse_kernel<B, 1>, at, bytes)) != cudaSuccess) return e;
    if ((e = cudaFuncSetAttribute(coop::fsr_coop_rows_kernel<B>, at, bytes)) != cudaSuccess) return e;
    return cudaFuncSetAttribute(coop::fsr_coop_reuse_kernel<B, kReuseSegs>, at, bytes);
}

template <int B>
cudaError_t launch_rows_b(const coop::RowsArgs& a, int wanted, int sm_count, cudaStream_t stream) {
    const size_t smem = sizeof(coop::Smem<4>);
    int grid = 0;
    cudaError_t e = persistent_grid(coop::fsr_coop_rows_kernel<B>, 4, smem, (long long)wanted * 4,
                                    sm_count, &grid);
    if (e != cudaSuccess) return e;
    coop::fsr_coop_rows_kernel<B><<<grid, coop::Cfg<4>::T, smem, stream>>>(a);
    return cudaGetLastError();
}

template <int B>
cudaError_t launch_b(const BatchArgs& a, const ImageArgs* one, cudaStream_t stream) {
    const size_t smem = sizeof(coop::Smem<4>);
    if (one) coop::fsr_coop_kernel<B, 4, true><<<(unsigned)a.total, coop::Cfg<4>::T, smem, stream>>>(a, *one);
    else coop::fsr_coop_kernel<B, 4, false><<<(unsigned)a.total, coop::Cfg<4>::T, smem, stream>>>(a, ImageArgs());
    return cudaGetLastError();
}

template <int B, int NSEG>
cudaError_t launch_reuse_n(const ReuseLaunchN<NSEG>& a, cudaStream_t stream) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)a.total);
    cfg.blockDim = dim3(coop::Cfg<4>::T);
    cfg.dynamicSmemBytes = sizeof(coop::Smem<4>);
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, coop::fsr_coop_reuse_kernel<B, NSEG>, a);
}

template <int B>
cudaError_t launch_reuse_b(const ReuseLaunch& a, cudaStream_t stream) {
    return a.nseg == 1 ? launch_reuse_n<B, 1>(one_image(a), stream) : launch_reuse_n<B, kReuseSegs>(a, stream);
}

}  // namespace

cudaError_t configure_coop() {
    cudaError_t e = configure_coop2();
    if (e != cudaSuccess) return e;
    if ((e = configure_b<2>()) != cudaSuccess) return e;
    if ((e = configure_b<4>()) != cudaSuccess) return e;
    if ((e = configure_b<8>()) != cudaSuccess) return e;
    return configure_b<16>();
}

cudaError_t launch_coop(const BatchArgs& a, int B, const ImageArgs* one, int sm_count, cudaStream_t stream) {
    if (a.total > (long long)kCoop4BlocksPerSm * sm_count) return launch_coop2(a, B, one, stream);
    switch (B) {
        case 2: return launch_b<2>(a, one, stream);
        case 4: return launch_b<4>(a, one, stream);
        case 8: return launch_b<8>(a, one, stream);
        case 16: return launch_b<16>(a, one, stream);
        default: return cudaErrorInvalidValue;
    }
}

size_t coop_rows_bytes() { return sizeof(unsigned long long) * (coop::kRowRing + 2); }

// A block with `iters` iterations takes up to 0.5 us for each beside three others
// on its SM (0.2 us alone): eight times that, and two seconds.
unsigned long long row_limit_ns(unsigned long long base_ns, int iters) {
    return (base_ns ? base_ns : 2000000000ull) + 4000ull * (unsigned long long)(iters + 16);
}

cudaError_t launch_coop_rows(const MethodArgs& mth, float delta, int n, const ImageArgs* ims, void* ring,
                             unsigned* status, unsigned long long* empty, int B, int sm_count, RowWaitHook hook,
                             cudaStream_t stream) {
    coop::RowsArgs a = {};
    a.mth = mth;
    a.delta = delta;
    a.lag = (mth.L + B - 1) / B + 1;
    a.ring = static_cast<unsigned long long*>(ring);
    a.status = status;
    a.empty = empty;
    a.n = n;
    int order[coop::kRowImages], iters = 0;
    for (int i = 0; i < n; ++i) order[i] = i;
    std::stable_sort(order, order + n, [&](int x, int y) { return ims[x].H > ims[y].H; });
    for (int i = 0; i < n; ++i) {
        a.im[i] = ims[order[i]];
        a.nby[i] = (a.im[i].H + B - 1) / B;
        a.rows += a.nby[i];
        iters = std::max(iters, a.im[i].K);
    }
    a.limit_ns = row_limit_ns(hook.base_ns, iters);
    const int wanted = (int)coop_rows_parallel(n, ims, mth.L, B);
    cudaError_t e = cudaMemsetAsync(ring, 0, coop_rows_bytes(), stream);
    if (e == cudaSuccess && hook.skip_row)   // the row counter starts at 1: nobody takes row 0
        e = cudaMemsetAsync(a.ring + coop::kRowRing, 1, 1, stream);
    if (e != cudaSuccess) return e;
    switch (B) {
        case 2: return launch_rows_b<2>(a, wanted, sm_count, stream);
        case 4: return launch_rows_b<4>(a, wanted, sm_count, stream);
        case 8: return launch_rows_b<8>(a, wanted, sm_count, stream);
        case 16: return launch_rows_b<16>(a, wanted, sm_count, stream);
        default: return cudaErrorInvalidValue;
    }
}

long long coop_rows_parallel(int n, const ImageArgs* ims, int L, int B) {
    const int lag = (L + B - 1) / B + 1;
    long long p = 0, rows = 0;
    for (int i = 0; i < n; ++i) {
        const long long nby = (ims[i].H + B - 1) / B;
        p += std::min<long long>(nby, ims[i].nbx / lag + 1);
        rows += nby;
    }
    return n <= coop::kRowImages && rows <= 0x7fffffffll ? p : 0x7fffffffll;
}

cudaError_t launch_coop_reuse(const ReuseLaunch& a, int B, cudaStream_t stream) {
    switch (B) {
        case 2: return launch_reuse_b<2>(a, stream);
        case 4: return launch_reuse_b<4>(a, stream);
        case 8: return launch_reuse_b<8>(a, stream);
        case 16: return launch_reuse_b<16>(a, stream);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace fsrk
