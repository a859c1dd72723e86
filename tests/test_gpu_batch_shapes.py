"""Launch shapes of batches. Shapes that the environment or single-problem tuning has set stay as they
are; the others rise where a size has many bands (the batch's geometries are read through the library's
own header)."""
import ctypes
import multiprocessing
import subprocess

import pytest

import ibdl_inputs as I

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

SOURCE = r"""
#include "ibdl_internal.cuh"
extern "C" void shape(void* batch, int i, int pi, int* out) {
  const ibdl::Geometry* g = (*static_cast<ibdl::Batch**>(batch))->geoms[i];  // ibdl_batch holds a Batch*
  out[0] = g->rows_per_cta[pi];
  out[1] = g->cols_per_cta[pi];
  out[2] = g->threads[pi];
}
"""


@pytest.fixture(scope="module")
def shape(tmp_path_factory):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2210_07403_gb300 import build as b

    d = tmp_path_factory.mktemp("shape")
    (d / "shape.cu").write_text(SOURCE)
    out = str(d / "libshape.so")
    subprocess.run([b._nvcc(), *b.ARCH, *b.FLAGS, "-I", b.CSRC, "-shared", "-o", out, str(d / "shape.cu"), b.LIB,
                    "-Xlinker", f"-rpath={b.PKG}"], check=True)
    lib = ctypes.CDLL(out)

    def read(B, i, pi):
        v = (ctypes.c_int * 3)()
        lib.shape(B._h, i, pi, v)
        return list(v)

    read.path = out
    return read


def _problems(count, sizes, pde="scalar", dipole="analytic", lams=(0.0,)):
    out = []
    for i in range(count):
        N = sizes[i % len(sizes)]
        bd = I.ellipse(N + 3 + i % 7, 0.22 + 0.001 * (i % 11), 0.3, rot=0.1 * i)
        out.append(I.Problem(f"p{i}", 2, N, 1.0, (0.0, 0.0), bd, None, pde, lam=lams[i % len(lams)], delta="cos",
                             dipole=dipole, symbol="spectral"))
    return out


@pytest.mark.parametrize("count", [2, 40])  # 40 problems of 32²: about 480 bands of two rows
def test_environment_shapes_reach_batches(shape, monkeypatch, count):
    from paper_2210_07403_gb300.ibdl import Batch

    def shapes():
        B = Batch(_problems(count, (32,)))
        s = [shape(B, 0, pi) for pi in range(3)]
        B.close()
        return s

    default = shapes()
    assert all(s[2] == 256 for s in default)
    if count == 40:
        assert all(s[0] > 2 for s in default)
    monkeypatch.setenv("IBDL_PLAN_R", "2")
    rows = shapes()
    assert [s[0] for s in rows] == [2, 2, 2] and [s[1:] for s in rows] == [s[1:] for s in default]
    monkeypatch.delenv("IBDL_PLAN_R")
    monkeypatch.setenv("IBDL_PLAN_C", "1")
    cols = shapes()
    assert [s[1] for s in cols] == [1, 1, 1] and [s[::2] for s in cols] == [s[::2] for s in default]
    monkeypatch.delenv("IBDL_PLAN_C")
    monkeypatch.setenv("IBDL_THREADS", "128")
    threads = shapes()
    assert [s[2] for s in threads] == [128, 128, 128] and [s[:2] for s in threads] == [s[:2] for s in default]


def _tuned(path, count):
    """(child process) the tuned shapes of a geometry and those of a batch's first and last problem"""
    from paper_2210_07403_gb300 import Geometry
    from paper_2210_07403_gb300.ibdl import Batch

    probs = _problems(count, (16,))
    g = Geometry.from_problem(probs[0])
    g.autotune()
    B = Batch(probs)
    lib = ctypes.CDLL(path)
    out = []
    for pi, precision in enumerate(("fp64", "fp32", "fp32x2")):
        plan = g.launch_plan(precision)
        row = [[plan["rows"], plan["cols"], plan["threads"]]]
        for i in (0, count - 1):
            v = (ctypes.c_int * 3)()
            lib.shape(B._h, i, pi, v)
            row.append(list(v))
        out.append(row)
    return out


@pytest.mark.parametrize("count", [2, 100])  # 100 problems of 16²: some 600 bands of two rows
def test_tuned_shapes_reach_batches(shape, count):
    # tuning holds for a process: in a child, so that no other test sees it
    with multiprocessing.get_context("spawn").Pool(1) as pool:
        for tuned, first, last in pool.apply(_tuned, (shape.path, count)):
            assert first == tuned and last == tuned
