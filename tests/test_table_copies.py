"""Tables copied from host vectors must be on the device before work on any stream reads them. A plain
cudaMemcpy from pageable memory does not promise that (it may return early and is ordered with the legacy stream
only), so no source uses one towards the device: copies are asynchronous on a named stream."""
import os
import re

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2210_07403_gb300", "csrc")


def test_no_unordered_copies_to_the_device():
    found = []
    for f in sorted(os.listdir(CSRC)):
        if f.endswith((".cu", ".cuh")):
            src = open(os.path.join(CSRC, f), encoding="utf-8").read()
            found += [(f, m.group(0)) for m in re.finditer(r"cudaMemcpy\s*\([^;]*HostToDevice", src)]
    assert not found


@pytest.mark.gpu
@pytest.mark.parametrize("dim,N,M", [(2, 512, 900), (3, 64, 3000)])
def test_first_application_on_a_side_stream(dim, N, M):
    """created and applied on a non-blocking stream with nothing between; 1e-12 as in test_gpu_parity.py"""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import ibdl_inputs as I
    from oracle import ibdl_oracle as O
    from paper_2210_07403_gb300 import Geometry

    b = I.fibonacci_sphere(M) if dim == 3 else I.star(M)
    og = O.Geometry(O.Grid(dim, N), b.X, b.n, b.w, "cos", "analytic", "spectral", "scalar", 0.0, 1.0, "dirichlet")
    q = np.random.default_rng(N).standard_normal(M)
    want = O.apply(og, q)
    qd = torch.from_numpy(q).cuda()
    torch.cuda.synchronize()
    s = torch.cuda.Stream()
    for _ in range(5):
        with torch.cuda.stream(s):
            g = Geometry(b.X, b.n, b.w, N)
            y = g.apply(qd)
        s.synchronize()
        assert np.abs(y.cpu().numpy() - want).max() < 1e-12 * np.abs(want).max()
        g.close()
