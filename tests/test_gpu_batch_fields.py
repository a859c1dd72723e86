"""Applications of batches whose operators hold several fields, on both sides of the threshold above which
a size's launch shapes rise (304 touched bands): every problem against the FP64 oracle, with mixed grid sizes,
λ = 0 and λ > 0, with the tolerances of test_gpu_parity.py."""
import numpy as np
import pytest

import ibdl_inputs as I
from oracle import ibdl_oracle as O

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _problems(count, sizes, pde="scalar", dipole="analytic", lams=(0.0,)):
    out = []
    for i in range(count):
        N = sizes[i % len(sizes)]
        bd = I.ellipse(N + 3 + i % 7, 0.22 + 0.001 * (i % 11), 0.3, rot=0.1 * i)
        out.append(I.Problem(f"p{i}", 2, N, 1.0, (0.0, 0.0), bd, None, pde, lam=lams[i % len(lams)], delta="cos",
                             dipole=dipole, symbol="spectral"))
    return out


@pytest.mark.parametrize("count", [4, 120])  # with 120 problems each size has 40 · 9 (16²) bands or more
@pytest.mark.parametrize("pde,dipole", [("stokes", "analytic"), ("stokes", "spectral_div"), ("scalar", "spectral_div")])
def test_multi_field_batches(pde, dipole, count):
    from paper_2210_07403_gb300.ibdl import Batch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    probs = _problems(count, (16, 32, 64), pde, dipole, lams=(0.0, 3.0))
    B = Batch(probs)
    q = np.random.default_rng(count).standard_normal(B.total)
    qd = torch.from_numpy(q).cuda()
    want = [O.apply(O.geometry_from_problem(p), q[B.offsets[b]:B.offsets[b + 1]]) for b, p in enumerate(probs)]
    for precision, tol in (("fp64", 1e-12), ("fp32x2", 1e-12), ("fp32", 2e-5)):
        y = B.apply(qd, precision=precision).cpu().numpy()
        for b in range(count):
            d = np.abs(y[B.offsets[b]:B.offsets[b + 1]] - want[b])
            assert np.linalg.norm(d) < tol * np.linalg.norm(want[b]) and d.max() < tol * np.abs(want[b]).max()
    B.close()
