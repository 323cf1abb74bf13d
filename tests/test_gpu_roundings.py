"""The binary32 arithmetic that two kernels share (the CTA-per-block kernel gives
the bits of the one-warp kernel) is written out rounding by rounding: compiled
with and without the compiler's own contraction of products and sums, the
transforms of both kernels and the weights give one result."""
import concurrent.futures
import ctypes
import os
import subprocess

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

PROBE = r"""
#include "fsr_coop.cuh"
using namespace fsrk;

__global__ void whole(const float2* in, float2* out) {   // a lane per column, 32 points each
    float re[32], im[32];
    for (int m = 0; m < 32; ++m) {
        re[m] = in[m * 32 + threadIdx.x].x;
        im[m] = in[m * 32 + threadIdx.x].y;
    }
    fft32<float>(re, im);
    for (int m = 0; m < 32; ++m) out[m * 32 + threadIdx.x] = make_float2(re[m], im[m]);
}

template <int N>
__global__ void split(const float2* in, float2* out) {
    using C = coop::Cfg<N>;
    __shared__ float2 X[S * coop::AS], cs[S];
    const int lane = threadIdx.x & 31, q = threadIdx.x >> 5;
    const int q2 = N == 4 ? ((q & 1) << 1) | (q >> 1) : q;
    if (threadIdx.x < S) cs[threadIdx.x] = make_float2(float(cos_2pi32(threadIdx.x)), float(sin_2pi32(threadIdx.x)));
    __syncthreads();
    float2 x[C::PTS], e[C::TT][N];
    for (int i = 0; i < C::PTS; ++i) x[i] = in[coop::in_index<N>(q2, i) * 32 + lane];
    coop::fft32_split<N>(x, e, X, cs, q, lane);
    for (int tt = 0; tt < C::TT; ++tt)
        for (int p = 0; p < N; ++p) out[(C::TT * q + tt + C::PTS * p) * 32 + lane] = e[tt][p];
}

__global__ void weights(float2* out) {   // w_f
    MethodArgs m = {};
    m.freq_weight = 1;
    for (int k = 0; k < 32; ++k) out[k * 32 + threadIdx.x] = make_float2(wf_value<float>(m, k, (int)threadIdx.x), 0.f);
}

extern "C" int run(int which, const void* in, void* out) {   // 1024 float2 each
    const float2* i = static_cast<const float2*>(in);
    float2* o = static_cast<float2*>(out);
    if (which == 0) whole<<<1, 32>>>(i, o);
    if (which == 1) split<4><<<1, 128>>>(i, o);
    if (which == 2) split<2><<<1, 64>>>(i, o);
    if (which == 3) weights<<<1, 32>>>(o);
    return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def probes(tmp_path_factory):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2202_13926_gb300 import build as b
    d = tmp_path_factory.mktemp("roundings")
    (d / "probe.cu").write_text(PROBE)

    def make(fmad):
        so = str(d / f"probe_{fmad}.so")
        subprocess.run([b._nvcc(), *b.ARCH, *b.NVCC_FLAGS, "-I", b.CSRC, f"-fmad={fmad}", "-shared",
                        str(d / "probe.cu"), "-o", so], check=True, capture_output=True, cwd=os.fspath(d))
        return ctypes.CDLL(so)
    with concurrent.futures.ThreadPoolExecutor(2) as ex:
        return list(ex.map(make, ("true", "false")))


def _run(lib, which, x):
    out = torch.zeros_like(x)
    torch.cuda.synchronize()
    assert lib.run(which, ctypes.c_void_p(x.data_ptr()), ctypes.c_void_p(out.data_ptr())) == 0
    return out


@pytest.mark.parametrize("seed", [1, 2, 3])
def test_transforms_do_not_depend_on_contraction(probes, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.randn(1024, 2, generator=g, device="cuda") * 100
    res = [_run(lib, which, x) for lib in probes for which in (0, 1, 2)]
    ref = torch.fft.fft(torch.view_as_complex(x.double()).view(32, 32), dim=0)
    got = torch.view_as_complex(res[0].double()).view(32, 32)
    assert (got - ref).abs().max() <= 5 * 2.0 ** -22 * ref.abs().max()   # five stages, each a few roundings
    for r in res[1:]:
        assert torch.equal(r, res[0])


def test_frequency_weight_does_not_depend_on_contraction(probes):
    x = torch.zeros(1024, 2, device="cuda")
    assert torch.equal(*(_run(lib, 3, x) for lib in probes))
