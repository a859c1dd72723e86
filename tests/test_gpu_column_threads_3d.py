"""The y and z passes of the 3-D operator take 64, 128 or 256 threads by grid size and precision, and with
them other column groups. Applications and transposes against the FP64 oracle at each size, for one and
three fields; 1e-12 as in test_gpu_parity.py."""
import numpy as np
import pytest

import ibdl_inputs as I
from oracle import ibdl_oracle as O

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _rel(a, b):
    d = np.abs(a - b)
    return float(max(np.linalg.norm(d) / np.linalg.norm(b), d.max() / np.abs(b).max()))


@pytest.mark.parametrize("dipole", ["analytic", "spectral_div"])
@pytest.mark.parametrize("N", [16, 32, 64, 128])
def test_column_threads(N, dipole):
    from paper_2210_07403_gb300 import Geometry

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    b = I.fibonacci_sphere(5 * N, 0.21, center=(0.47, 0.9, 0.55))  # across a face
    og = O.Geometry(O.Grid(3, N), b.X, b.n, b.w, "cos", dipole, "spectral", "scalar", 2.0, 1.0, "dirichlet")
    g = Geometry(b.X, b.n, b.w, N, pde="scalar", dipole=dipole, delta="cos", lam=2.0)
    q = np.random.default_rng(N).standard_normal(og.M)
    qd = torch.from_numpy(q).cuda()
    want, wt = O.apply(og, q), O.transpose_apply(og, q)
    for precision in ("fp64", "fp32x2"):
        assert _rel(g.apply(qd, precision=precision).cpu().numpy(), want) < 1e-12
        assert _rel(g.apply_transpose(qd, precision=precision).cpu().numpy(), wt) < 1e-12
    g.close()
