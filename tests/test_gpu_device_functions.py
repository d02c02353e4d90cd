"""The kernels' own elementary functions on the device (``-m gpu``), compiled
from the library's source into a probe: the packed float32 erfcx of the paired
short range (``test_gpu_erfc.py`` takes the scalar one) and the float64
reciprocal square root."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

PROBE = r"""
#include "k_short.cu"

// what else k_short.cu calls, never reached here
namespace bsw {
cudaError_t scan_exclusive(int*, int, int*, cudaStream_t, int*) { return cudaErrorNotSupported; }
void set_last_error(const char*) {}
void cheb_fit(const std::function<long double(long double)>&, long double, long double, int, double*, int) {}
}
using namespace bsw;

// out[0..n): erfcx_f; out[n..2n): erfcx_2 of neighbouring arguments, the last of an odd count with itself
__global__ void k_erfcx(int n, const float* x, float* out)
{
    const int i = 2 * (blockIdx.x * blockDim.x + threadIdx.x);
    if (i >= n) return;
    const bool two = i + 1 < n;
    const float2 v = upk2(erfcx_2(pk2(x[i], x[two ? i + 1 : i])));
    out[i] = erfcx_f(x[i]);
    out[n + i] = v.x;
    if (two) {
        out[i + 1] = erfcx_f(x[i + 1]);
        out[n + i + 1] = v.y;
    }
}

__global__ void k_rsqrt(int n, const double* a, double* out)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] = rsqrt_h(a[i]);
}

extern "C" int probe_erfcx(int n, const float* x, float* out)
{
    k_erfcx<<<(n + 511) / 512, 256>>>(n, x, out);
    return (int)cudaDeviceSynchronize();
}
extern "C" int probe_rsqrt(int n, const double* a, double* out)
{
    k_rsqrt<<<(n + 255) / 256, 256>>>(n, a, out);
    return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    from paper_2406_07366_gb300 import build as b
    d = tmp_path_factory.mktemp("probe")
    src, so = d / "probe.cu", d / "probe.so"
    src.write_text(PROBE)
    nvcc = b._nvcc()
    lib = b._cuda_lib_dir(nvcc)
    subprocess.run([nvcc, str(src), "-o", str(so), *b.ARCH, "-shared", "-O3", "-std=c++17", "-Xcompiler", "-fPIC",
                    "--expt-relaxed-constexpr", "-I", b.INCLUDE, "-I", b.CSRC, "-L", lib, "-lcudart", "-Xlinker",
                    "-rpath," + lib], check=True, capture_output=True, cwd=os.path.dirname(str(src)))
    torch.cuda.init()
    return ctypes.CDLL(str(so))


@pytest.mark.parametrize("n", [(0x40a00000 - 0x3f800000) + 1, 1000])
def test_packed_erfcx_against_cuda_and_the_scalar_form(probe, n):
    """exp(x^2) erfc(x) for every float32 d = 1 + x/2 in [1, 5], an odd count in
    pairs (and an even one): the error against CUDA's float64 erfcx is that of
    the scalar form and below the fit's 4e-7.  The reciprocals differ by at most
    one unit in the last place (Newton's step leaves 2^-46 and one rounding),
    2^-23 relative; |t p' / p| <= 2.3 makes that up to 4.6 units of the value,
    and the last three steps of the sum may round the other way: 8."""
    d = torch.arange(0x3f800000, 0x3f800000 + n, dtype=torch.int32, device="cuda").view(torch.float32)
    x = 2 * (d - 1)  # exact
    out = torch.empty(2 * n, dtype=torch.float32, device="cuda")
    torch.cuda.synchronize()
    assert probe.probe_erfcx(n, ctypes.c_void_p(x.data_ptr()), ctypes.c_void_p(out.data_ptr())) == 0
    exact = torch.special.erfcx(x.double())
    one, two = out[:n].double(), out[n:].double()
    e1, e2 = (one / exact - 1).abs(), (two / exact - 1).abs()
    ulp = 2.0 ** (torch.floor(torch.log2(one)) - 23)
    far = ((one - two).abs() / ulp).max()
    print(f"scalar max {e1.max():.3e} rms {e1.square().mean().sqrt():.4e}, packed max {e2.max():.3e} rms "
          f"{e2.square().mean().sqrt():.4e}, {int((one != two).sum())} of {n} differ, by at most {far:.1f} units")
    assert float(e1.max()) < 4e-7 and float(e2.max()) < 4e-7
    assert float(e2.square().mean()) <= 1.02 * float(e1.square().mean())
    assert float(far) <= 8


def test_reciprocal_square_root_within_its_bound(probe):
    """y = rsqrt_h(a) over sixty decades and densely over [1, 4): the error
    (1 - a y^2) / 2, formed exactly enough in extended precision.  The product
    a y in the residual and the last step round by 2^-53 each, the first at half
    weight: 1.5 * 2^-53, what the iteration leaves (2^-58) and second-order terms."""
    rng = np.random.default_rng(0)
    a = np.concatenate([10.0 ** rng.uniform(-30, 30, 1 << 20), 1 + 3 * rng.random(1 << 21), 1 + 3 * np.arange(1 << 16) / 2.0 ** 16,
                        2.0 ** np.arange(-200, 200), np.nextafter(2.0 ** np.arange(-200.0, 200.0), 0)])
    x = torch.from_numpy(a).cuda()
    out = torch.empty_like(x)
    torch.cuda.synchronize()
    assert probe.probe_rsqrt(len(a), ctypes.c_void_p(x.data_ptr()), ctypes.c_void_p(out.data_ptr())) == 0
    y = out.cpu().numpy().astype(np.longdouble)
    err = np.abs((1 - a.astype(np.longdouble) * y * y) / 2).astype(np.float64)
    lib = np.abs((1 - a.astype(np.longdouble) * torch.rsqrt(x).cpu().numpy().astype(np.longdouble) ** 2) / 2)
    print("rsqrt_h max %.3f 2^-53, CUDA's rsqrt %.3f" % (err.max() * 2.0 ** 53, float(lib.max()) * 2.0 ** 53))
    assert err.max() < 1.5 * 2.0 ** -53 + 2.0 ** -57
