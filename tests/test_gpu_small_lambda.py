"""A small screening λ > 0: the zero mode of the analytic dipole spread is zero in exact arithmetic
(each kernel's derivative weights sum to zero), so FP32 rounding in it must not be amplified by 1/λ.
FP32 applications stay within the λ = 1 tolerance of test_gpu_parity.py (2e-5) at λ = 1e-4, where one
rounding error of the mean would be some 1e-2."""
import numpy as np
import pytest

import ibdl_inputs as I
from oracle import ibdl_oracle as O

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("dim,pde,N,M", [(2, "scalar", 64, 100), (2, "scalar", 256, 403), (2, "stokes", 128, 201), (3, "scalar", 32, 700)])
def test_small_lambda(dim, pde, N, M):
    from paper_2210_07403_gb300 import Geometry

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    b = I.fibonacci_sphere(M) if dim == 3 else I.star(M)
    og = O.Geometry(O.Grid(dim, N), b.X, b.n, b.w, "cos", "analytic", "spectral", pde, 1e-4, 1.0, "dirichlet")
    g = Geometry(b.X, b.n, b.w, N, pde=pde, lam=1e-4)
    q = np.random.default_rng(N).standard_normal(og.ncomp * M)
    # the oracle's field without its mean, which is its own FP64 rounding amplified by 1/λ
    u = O.grid_field(og, q).reshape((og.ncomp,) + (N,) * dim)
    want = np.concatenate([O.interp(og, v - v.mean()) for v in u]) + 0.5 * q
    for precision, tol in (("fp64", 1e-12), ("fp32", 2e-5)):
        got = g.apply(torch.from_numpy(q).cuda(), precision=precision).cpu().numpy()
        assert np.linalg.norm(got - want) / np.linalg.norm(want) < tol
        assert np.abs(got - want).max() / np.abs(want).max() < tol
    # a source term keeps its mean: u_g of a constant source is −1/λ
    src = torch.ones((og.ncomp,) + (N,) * dim, dtype=torch.float64, device="cuda")
    u = g.evaluate_field(torch.zeros(og.ncomp * M, dtype=torch.float64, device="cuda"), g=src)
    assert torch.allclose(u, torch.full_like(u, -1e4), rtol=1e-12)
    g.close()
