"""Row transforms are run only for the rows that some point's stencil meets. Against the FP64
oracle: boundaries that meet few rows, rows across the periodic edge, rows with gaps between them
and every row, at several band heights, with the spectra of all other rows left full of NaN by an
earlier field evaluation (they must not be read). Tolerances as in test_gpu_parity.py: 1e-12 in FP64
and float-float, 2e-5 in FP32 (relative 2-norm and element-wise)."""
import numpy as np
import pytest

import ibdl_inputs as I
from oracle import ibdl_oracle as O

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

TOL = {"fp64": 1e-12, "fp32": 2e-5, "fp32x2": 1e-12}


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2210_07403_gb300 import build as b
    from paper_2210_07403_gb300 import ibdl

    b.build()
    ibdl.load()


def _rel(a, b):
    a, b = np.asarray(a, dtype=np.float64), np.asarray(b, dtype=np.float64)
    d = np.abs(a - b)
    return float(max(np.linalg.norm(d) / np.linalg.norm(b), d.max() / np.abs(b).max()))


def _join(*bds):
    return (np.concatenate([b.X for b in bds], axis=1), np.concatenate([b.n for b in bds], axis=1),
            np.concatenate([b.w for b in bds]))


def _boundary(kind, N):
    h = 1.0 / N
    if kind == "one_point":
        return np.array([[0.3], [0.6]]), np.array([[0.6], [0.8]]), np.array([h])
    if kind == "edge":  # across y = 0 and x = 0
        b = I.circle(40, 3.0 * h, (0.01, 1.0 - 0.7 * h))
    elif kind == "flat":
        b = I.ellipse(2 * N, 0.4, 1.5 * h)
    elif kind == "gaps":
        return _join(I.circle(31, 2.0 * h, (0.5, 0.15)), I.circle(50, 2.5 * h, (0.2, 0.71)))
    else:  # every row
        b = I.ellipse(3 * N, 0.2, 0.497)
    return b.X, b.n, b.w


@pytest.mark.parametrize("rows", [2, 4, 8])
@pytest.mark.parametrize("kind", ["one_point", "edge", "flat", "gaps", "tall"])
@pytest.mark.parametrize("N,pde,dipole,split", [(16, "scalar", "analytic", 0), (64, "scalar", "spectral_div", 0),
                                                (64, "stokes", "analytic", 0), (128, "stokes", "spectral_div", 1),
                                                (512, "stokes", "analytic", 0)])
def test_touched_rows_2d(N, pde, dipole, split, kind, rows, monkeypatch):
    from paper_2210_07403_gb300 import Geometry

    monkeypatch.setenv("IBDL_PLAN_R", str(rows))
    if split:
        monkeypatch.setenv("IBDL_SPLIT_FIELDS", "1")
    X, n, w = _boundary(kind, N)
    og = O.Geometry(O.Grid(2, N), X, n, w, "cos", dipole, "spectral", pde, 0.0, 1.0, "dirichlet")
    g = Geometry(X, n, w, N, pde=pde, dipole=dipole)
    rng = np.random.default_rng(N + rows)
    q = rng.standard_normal(og.ncomp * og.M)
    qd = torch.from_numpy(q).cuda()
    bad = torch.full_like(qd, float("nan"))
    want = O.apply(og, q)
    wantT = None
    if pde == "scalar":
        wantT = O.transpose_apply(og, q)
    elif dipole == "analytic":
        wantT = O.stokes_transpose_apply(og, q)
    for precision in ("fp64", "fp32", "fp32x2"):
        assert torch.isnan(g.evaluate_field(bad)).all()
        assert _rel(g.apply(qd, precision=precision).cpu().numpy(), want) < TOL[precision]
        assert torch.isnan(g.apply(bad, precision=precision)).all()
        if wantT is not None:
            assert _rel(g.apply_transpose(qd, precision=precision).cpu().numpy(), wantT) < TOL[precision]
    field = O.grid_field(og, q)
    assert _rel(g.evaluate_field(qd).cpu().numpy(), field) < 1e-12
    g.close()


def _surface(kind, N):
    h = 1.0 / N
    if kind == "one_point":
        return np.array([[0.3], [0.6], [0.9]]), np.array([[0.6], [0.8], [0.0]]), np.array([h * h])
    if kind == "edge":  # across y = 0 and z = 0
        b = I.fibonacci_sphere(60, 2.0 * h, (0.4, 1.0 - 0.3 * h, 0.2 * h))
    elif kind == "gaps":
        return _join(I.fibonacci_sphere(50, 1.6 * h, (0.5, 0.2, 0.2)), I.fibonacci_sphere(70, 2.2 * h, (0.5, 0.75, 0.7)))
    else:  # every plane
        b = I.fibonacci_sphere(6 * N * N, 0.499)
    return b.X, b.n, b.w


@pytest.mark.parametrize("rows", [2, 8])
@pytest.mark.parametrize("kind", ["one_point", "edge", "gaps", "tall"])
@pytest.mark.parametrize("N,dipole", [(16, "analytic"), (32, "spectral_div"), (64, "analytic")])
def test_touched_rows_3d(N, dipole, kind, rows, monkeypatch):
    from paper_2210_07403_gb300 import Geometry

    monkeypatch.setenv("IBDL_PLAN3_R", str(rows))
    X, n, w = _surface(kind, N)
    og = O.Geometry(O.Grid(3, N), X, n, w, "cos", dipole, "spectral", "scalar", 0.0, 1.0, "dirichlet")
    g = Geometry(X, n, w, N, dipole=dipole)
    rng = np.random.default_rng(N + rows)
    q = rng.standard_normal(og.M)
    qd = torch.from_numpy(q).cuda()
    bad = torch.full_like(qd, float("nan"))
    want, wantT = O.apply(og, q), O.transpose_apply(og, q)
    for precision in ("fp64", "fp32", "fp32x2"):
        assert torch.isnan(g.evaluate_field(bad)).all()
        assert _rel(g.apply(qd, precision=precision).cpu().numpy(), want) < TOL[precision]
        assert torch.isnan(g.apply(bad, precision=precision)).all()
        assert _rel(g.apply_transpose(qd, precision=precision).cpu().numpy(), wantT) < TOL[precision]
    assert _rel(g.evaluate_field(qd).cpu().numpy(), O.grid_field(og, q)) < 1e-12
    g.close()
