"""The quotients of the Fourier symbols are the correctly rounded ones to the last bit, in FP64 and (3-D)
in FP32: the device functions compiled into small kernels, against numpy's division."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

SOURCE = r"""
#include "apply2d_kernels.cuh"
#include "apply3d_kernels.cuh"
using namespace ibdl;
template <typename T>
__global__ void k_symbol3(int n, const T* lap, T lam, T scale, T* out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const T lap1[2] = {lap[i], T(0)}, der1[2] = {T(0), T(0)};
  const cplx<T> in[1] = {mk(T(1), T(0))};
  cplx<T> o[3];
  symbol3<T, OP3_SCALAR_AN>(lap1, der1, lam, scale, 0, 0, 1, 1, in, o);
  out[i] = o[0].x;
}
extern "C" int symbol3_f32(int n, const float* lap, float lam, float scale, float* out) {
  k_symbol3<float><<<(n + 255) / 256, 256>>>(n, lap, lam, scale, out);
  return (int)cudaDeviceSynchronize();
}
extern "C" int symbol3_f64(int n, const double* lap, double lam, double scale, double* out) {
  k_symbol3<double><<<(n + 255) / 256, 256>>>(n, lap, lam, scale, out);
  return (int)cudaDeviceSynchronize();
}
__global__ void k_quotient(int n, const double* a, const double* b, double* out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) out[i] = sym_div(a[i], b[i]);
}
extern "C" int quotient_f64(int n, const double* a, const double* b, double* out) {
  k_quotient<<<(n + 255) / 256, 256>>>(n, a, b, out);
  return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2210_07403_gb300 import build as b

    d = tmp_path_factory.mktemp("symbol")
    (d / "symbol.cu").write_text(SOURCE)
    out = str(d / "libsymbol.so")
    subprocess.run([b._nvcc(), *b.ARCH, *b.FLAGS, "-I", b.CSRC, "-shared", "-o", out, str(d / "symbol.cu"),
                    os.path.join(b.PKG, "libibdl.so"), "-Xlinker", f"-rpath={b.PKG}"], check=True)
    torch.zeros(1, device="cuda")
    return ctypes.CDLL(out)


@pytest.mark.parametrize("n", [16, 128, 256])
@pytest.mark.parametrize("dtype", [np.float32, np.float64])
def test_symbol3_is_rounded(lib, dtype, n):
    rng = np.random.default_rng(n)
    lap = (4 * np.pi ** 2 * rng.uniform(0, 3 * (n / 2) ** 2, size=100000)).astype(dtype)
    scale = dtype(0.5 / n ** 3)
    d = torch.from_numpy(lap).cuda()
    out = torch.empty_like(d)
    f, c = (lib.symbol3_f32, ctypes.c_float) if dtype == np.float32 else (lib.symbol3_f64, ctypes.c_double)
    for lam in (dtype(0.0), dtype(0.37), dtype(40.0)):
        assert f(len(lap), ctypes.c_void_p(d.data_ptr()), c(lam), c(scale), ctypes.c_void_p(out.data_ptr())) == 0
        assert np.array_equal(out.cpu().numpy(), scale / (lap + lam))


def test_fp64_quotient_is_rounded(lib):
    """every exponent of the divisor, subnormal numbers included, and quotients that over- and underflow"""
    rng = np.random.default_rng(1)
    b = rng.integers(1, 0x7FF0000000000000, size=200000, dtype=np.int64).view(np.float64)
    a = np.ldexp(rng.uniform(0.5, 1.0, size=b.size), rng.integers(-60, 61, size=b.size))
    da, db = torch.from_numpy(a).cuda(), torch.from_numpy(b).cuda()
    out = torch.empty_like(da)
    assert lib.quotient_f64(b.size, *(ctypes.c_void_p(t.data_ptr()) for t in (da, db, out))) == 0
    with np.errstate(over="ignore", under="ignore"):
        assert np.array_equal(out.cpu().numpy(), a / b)
