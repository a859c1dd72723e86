"""Small grids run FP64 and float-float kernels with two or four elements per lane. Applications,
transposes and fields against the FP64 oracle at every such size, for one to four fields, with two-row
bands and single columns (few elements) and with taller bands (the ordinary kernels); 1e-12 as in
test_gpu_parity.py."""
import numpy as np
import pytest

import ibdl_inputs as I
from oracle import ibdl_oracle as O

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _rel(a, b):
    d = np.abs(a - b)
    return float(max(np.linalg.norm(d) / np.linalg.norm(b), d.max() / np.abs(b).max()))


@pytest.mark.parametrize("rows", [2, 4])
@pytest.mark.parametrize("pde,dipole", [("scalar", "analytic"), ("scalar", "spectral_div"), ("stokes", "analytic"),
                                        ("stokes", "spectral_div")])
@pytest.mark.parametrize("N", [16, 32, 64, 128, 256, 512, 1024])
def test_few_elements(N, pde, dipole, rows, monkeypatch):
    from paper_2210_07403_gb300 import Geometry

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    monkeypatch.setenv("IBDL_PLAN_R", str(rows))
    b = I.star(int(1.3 * N) + 5, 0.21, center=(0.47, 0.9))  # across the edge
    og = O.Geometry(O.Grid(2, N), b.X, b.n, b.w, "sqrt", dipole, "spectral", pde, 2.0, 1.0, "dirichlet")
    g = Geometry(b.X, b.n, b.w, N, pde=pde, dipole=dipole, delta="sqrt", lam=2.0)
    q = np.random.default_rng(N).standard_normal(og.ncomp * og.M)
    qd = torch.from_numpy(q).cuda()
    want = O.apply(og, q)
    for precision in ("fp64", "fp32x2"):
        assert _rel(g.apply(qd, precision=precision).cpu().numpy(), want) < 1e-12
        if pde == "scalar" or dipole == "analytic":
            wt = O.transpose_apply(og, q) if pde == "scalar" else O.stokes_transpose_apply(og, q)
            assert _rel(g.apply_transpose(qd, precision=precision).cpu().numpy(), wt) < 1e-12
    assert _rel(g.evaluate_field(qd).cpu().numpy(), O.grid_field(og, q)) < 1e-12
    g.close()
