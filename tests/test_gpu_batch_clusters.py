"""Batched solves on both sides of the Arnoldi step's cluster size (clusters of four CTAs per problem
up to 32 problems, of two beyond): every problem against the FP64 oracle. Point counts differ, so the last
CTA of a cluster holds slices of every length. The operators' condition numbers are at most 1.8, so at
relative residual 1e-10 the largest element's error stays below 1e-10 · 1.8 · √49 < 2e-9 of the largest."""
import numpy as np
import pytest

import ibdl_inputs as I
from oracle import ibdl_oracle as O

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _rel(a, b):
    d = np.abs(a - b)
    return float(max(np.linalg.norm(d) / np.linalg.norm(b), d.max() / np.abs(b).max()))


@pytest.mark.parametrize("count", [32, 33])
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_batch_solve_cluster_sizes(count, precision):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2210_07403_gb300.ibdl import Batch

    rng = np.random.default_rng(9)
    probs = []
    for i in range(count):
        bd = I.ellipse(17 + i, 0.2, 0.27, rot=0.1 * i)
        Ub = I.random_modes(bd.t, 4, 1.0, rng, 1, decay=True)
        probs.append(I.Problem(f"p{i}", 2, 32, 1.0, (0.0, 0.0), bd, Ub, "scalar", lam=1.0 + i, delta="cos",
                               dipole="analytic", symbol="spectral"))
    B = Batch(probs)
    ub = torch.from_numpy(np.concatenate([p.Ub.reshape(-1) for p in probs])).cuda()
    Q, infos, st = B.solve(ub, rtol=1e-10, precision=precision)
    assert st == 0
    Q = Q.cpu().numpy()
    for b, p in enumerate(probs):
        sl = slice(B.offsets[b], B.offsets[b + 1])
        assert infos[b]["rel_residual"] <= 1e-10
        assert _rel(Q[sl], O.solve(O.geometry_from_problem(p), p.Ub, 1e-12).x) < 2e-9
