"""FP64 transforms of data near the top of the FP64 range: no twiddle form may multiply a value by more than
the tangent of its angle (below n/6), so data that overflow nowhere in the operator itself must not overflow
in its butterflies. Densities of size 2⁹⁶⁰ (1e289; the spread's weights of up to 0.4·w/h³ and the transforms'
sums stay below 2³⁵) against the same density of size 1 on the same geometry: scaling by a power of two is
exact, so only the order of the atomic additions differs (1e-12 as in test_gpu_parity.py). The grids cover every
form of the transform: two elements per lane, eight, and the radix-2 and radix-4 tails, in 2-D, 3-D and
batches."""
import numpy as np
import pytest

import ibdl_inputs as I

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

BIG = 2.0 ** 960


def _rel(a, b):
    d = np.abs(a - b)
    return float(max(np.linalg.norm(d) / np.linalg.norm(b), d.max() / np.abs(b).max()))


@pytest.mark.parametrize("dim,N", [(2, 16), (2, 128), (2, 256), (2, 512), (2, 1024), (2, 2048), (3, 16), (3, 64), (3, 128)])
def test_large_densities(dim, N):
    from paper_2210_07403_gb300 import Geometry

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    b = I.fibonacci_sphere(N * N // 2) if dim == 3 else I.star(int(1.3 * N))
    g = Geometry(b.X, b.n, b.w, N, lam=1.0)
    q = torch.from_numpy(np.random.default_rng(N).standard_normal(g.nd)).cuda()
    big = q * BIG
    assert _rel((g.apply(big) / BIG).cpu().numpy(), g.apply(q).cpu().numpy()) < 1e-12
    assert _rel((g.apply_transpose(big) / BIG).cpu().numpy(), g.apply_transpose(q).cpu().numpy()) < 1e-12
    assert _rel((g.evaluate_field(big) / BIG).cpu().numpy(), g.evaluate_field(q).cpu().numpy()) < 1e-12
    g.close()


def test_large_densities_batch():
    from paper_2210_07403_gb300.ibdl import Batch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    probs = [I.Problem(f"p{i}", 2, N, 1.0, (0.0, 0.0), I.ellipse(N + 5, 0.2, 0.27), None, "scalar", lam=1.0, delta="cos",
                       dipole="analytic", symbol="spectral") for i, N in enumerate((16, 32, 64, 128, 256))]
    B = Batch(probs)
    q = torch.from_numpy(np.random.default_rng(1).standard_normal(B.total)).cuda()
    a, b = (B.apply(q * BIG) / BIG).cpu().numpy(), B.apply(q).cpu().numpy()
    for i in range(len(probs)):
        sl = slice(B.offsets[i], B.offsets[i + 1])
        assert _rel(a[sl], b[sl]) < 1e-12
    B.close()
