"""The quotient of the 3-D Fourier symbol, scale/(|k|² + λ), is the correctly rounded one in FP32, to the
last bit: the device function compiled into a small kernel, against numpy's division."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

SOURCE = r"""
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
def test_symbol3_is_rounded(lib, n):
    rng = np.random.default_rng(n)
    lap = (4 * np.pi ** 2 * rng.uniform(0, 3 * (n / 2) ** 2, size=100000)).astype(np.float32)
    scale = np.float32(0.5 / n ** 3)
    d = torch.from_numpy(lap).cuda()
    out = torch.empty_like(d)
    for lam in (np.float32(0.0), np.float32(0.37), np.float32(40.0)):
        assert lib.symbol3_f32(len(lap), ctypes.c_void_p(d.data_ptr()), ctypes.c_float(lam), ctypes.c_float(scale),
                               ctypes.c_void_p(out.data_ptr())) == 0
        assert np.array_equal(out.cpu().numpy(), scale / (lap + lam))
