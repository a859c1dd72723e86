"""Near-boundary interpolation by row segments, against the oracle on the same inputs: the smallest
grid (two rows per 32 nodes), a boundary with more points near a segment than the kernel collects at a
time, a curve across the periodic edges of a box with a shifted origin, and a mask with holes.
Tolerance 1e-12 of the largest value, as in test_gpu_postproc.py."""
import numpy as np
import pytest

import ibdl_inputs as I
from oracle import ibdl_oracle as O

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("N,M,R,centre,origin,m1", [
    (16, 40, 0.25, (0.5, 0.5), (0.0, 0.0), 2.5), (16, 7, 0.3, (0.1, 0.9), (0.0, 0.0), 1.0),
    (32, 60, 0.25, (0.02, 0.5), (-0.5, -0.25), 3.0), (64, 2000, 0.1, (0.5, 0.5), (0.0, 0.0), 4.0),
    (128, 3000, 0.3, (0.7, 0.05), (0.0, 0.0), 6.0), (256, 500, 0.2, (0.5, 0.96), (0.3, 0.7), 9.5)])
def test_near_boundary_segments(N, M, R, centre, origin, m1):
    from paper_2210_07403_gb300 import Geometry

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    b = I.circle(M, R, centre)
    og = O.Geometry(O.Grid(2, N, 1.0, origin), b.X, b.n, b.w)
    rng = np.random.default_rng(N + M)
    Ub, u = rng.standard_normal(M), rng.standard_normal((N, N))
    omega = rng.random((N, N)) < 0.8
    g = Geometry(b.X, b.n, b.w, N, origin=origin)
    out = g.near_boundary(torch.from_numpy(Ub), torch.from_numpy(u).cuda(), torch.from_numpy(omega), m1, m1 + 2)
    ref = O.near_boundary_interp(og, Ub, u, omega, m1, m1 + 2)
    assert np.abs(out.cpu().numpy() - ref).max() < 1e-12 * max(np.abs(u).max(), np.abs(Ub).max())
    assert not np.array_equal(ref, u)
    g.close()
