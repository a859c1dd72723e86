"""λ so small that it rounds to zero in FP32 (below 2⁻¹⁵⁰, about 7e-46): FP32 and float-float
applications drop the zero mode as for λ = 0, instead of dividing it by zero. Against the FP64 oracle
at λ = 0 for the operators whose zero mode carries nothing (a dipole spread or gather has no mean), 2e-5
in FP32 and 1e-12 in float-float as in test_gpu_parity.py; the single layer against its λ = 0 result in the
same arithmetic, 2e-5."""
import numpy as np
import pytest

import ibdl_inputs as I
from oracle import ibdl_oracle as O

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

TOL = {"fp32": 2e-5, "fp32x2": 1e-12}


def _rel(a, b):
    d = np.abs(a - b)
    return float(max(np.linalg.norm(d) / np.linalg.norm(b), d.max() / np.abs(b).max()))


@pytest.mark.parametrize("lam", [5e-324, 1e-46])
@pytest.mark.parametrize("dipole", ["analytic", "spectral_div"])
@pytest.mark.parametrize("dim,pde,N,M", [(2, "scalar", 64, 100), (2, "scalar", 512, 700), (2, "stokes", 64, 100),
                                         (3, "scalar", 16, 300), (3, "scalar", 64, 2000)])
def test_lambda_below_fp32(dim, pde, N, M, dipole, lam):
    from paper_2210_07403_gb300 import Geometry

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    b = I.fibonacci_sphere(M) if dim == 3 else I.star(M)
    og = O.Geometry(O.Grid(dim, N), b.X, b.n, b.w, "cos", dipole, "spectral", pde, 0.0, 1.0, "dirichlet")
    g = Geometry(b.X, b.n, b.w, N, pde=pde, dipole=dipole, lam=lam)
    q = np.random.default_rng(N).standard_normal(og.ncomp * M)
    qd = torch.from_numpy(q).cuda()
    for precision, tol in TOL.items():
        assert _rel(g.apply(qd, precision=precision).cpu().numpy(), O.apply(og, q)) < tol
        if pde == "scalar":
            assert _rel(g.apply_transpose(qd, precision=precision).cpu().numpy(), O.transpose_apply(og, q)) < tol
    if dim == 2 and pde == "scalar":
        g0 = Geometry(b.X, b.n, b.w, N, dipole=dipole)
        assert _rel(g.single_layer(qd, precision="fp32").cpu().numpy(), g0.single_layer(qd, precision="fp32").cpu().numpy()) < 2e-5
        g0.close()
    g.close()


@pytest.mark.parametrize("dipole", ["analytic", "spectral_div"])
def test_batch_lambda_below_fp32(dipole):
    from paper_2210_07403_gb300.ibdl import Batch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    probs = []
    for i, N in enumerate((16, 64, 32)):
        bd = I.ellipse(N + 9, 0.2, 0.27, rot=0.4 * i)
        probs.append(I.Problem(f"p{i}", 2, N, 1.0, (0.0, 0.0), bd, None, "scalar", lam=1e-46, delta="cos",
                               dipole=dipole, symbol="spectral"))
    B = Batch(probs)
    q = np.random.default_rng(6).standard_normal(B.total)
    for precision, tol in TOL.items():
        y = B.apply(torch.from_numpy(q).cuda(), precision=precision).cpu().numpy()
        for b, p in enumerate(probs):
            sl = slice(B.offsets[b], B.offsets[b + 1])
            og = O.Geometry(O.Grid(2, p.N), p.bd.X, p.bd.n, p.bd.w, "cos", dipole, "spectral", "scalar", 0.0, 1.0, "dirichlet")
            assert _rel(y[sl], O.apply(og, q[sl])) < tol
    B.close()
