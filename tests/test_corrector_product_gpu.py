"""M_i^-1 r of the FP32 corrector, whose factors are FP16 parts on the tensor cores, against 64 bits: no
further off than FP32 multiply-adds over FP32 rows of M_i^-1."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from inputs.voronoi import periodic_voronoi
from oracle.mesh import from_polymesh

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def product(tmp_path_factory):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2605_00619_gb300 import afe, build
    afe.lib()
    out = str(tmp_path_factory.mktemp("corrector") / "libcorrector_product.so")
    subprocess.run([build._nvcc(), "-O2", "-std=c++17", "-shared", "-Xcompiler", "-fPIC", "--expt-relaxed-constexpr",
                    *build.ARCH, "-I" + build.CSRC, "-I" + build.INCLUDE, "-I" + os.path.join(build.LIBDIR, "gen"),
                    os.path.join(HERE, "corrector_product.cu"), build.LIBPATH, "-Xlinker", "-rpath=" + build.LIBDIR,
                    "-o", out], check=True)
    fn = ctypes.CDLL(out).corrector_product
    ptr = np.ctypeslib.ndpointer
    fn.argtypes = [ctypes.c_int, ctypes.c_int64, ptr(np.int64), ptr(np.int64), ptr(np.float64), ptr(np.float32),
                   ptr(np.float64)]
    fn.restype = ctypes.c_int

    def run(N, minvs, rs):
        n = np.array([len(m) for m in minvs])
        ld = (n + 15) // 16 * 16 + 8
        node_ptr = np.concatenate([[0], np.cumsum(n)]).astype(np.int64)
        minv_ptr = np.concatenate([[0], np.cumsum((n * ld + 31) // 32 * 32)]).astype(np.int64)
        rows = np.zeros(minv_ptr[-1])
        for k, m in enumerate(minvs):
            rows[minv_ptr[k]:minv_ptr[k] + n[k] * ld[k]].reshape(n[k], ld[k])[:, :n[k]] = m
        du = np.empty((node_ptr[-1], 5))
        assert fn(N, len(n), node_ptr, minv_ptr, rows, np.ascontiguousarray(np.concatenate(rs)), du) == 0
        return np.split(du, node_ptr[1:-1])
    return run


def _fp32(minv, r):
    """FP32 multiply-adds in order over FP32 rows (the product of two FP32 values is exact in FP64)."""
    a = minv.astype(np.float32).astype(np.float64)
    acc = np.zeros(r.shape, np.float32)
    for k in range(len(a)):
        acc = (a[:, k:k + 1] * r[k].astype(np.float64) + acc).astype(np.float32)
    return acc


@pytest.mark.parametrize("kind", ["random", "smooth"])
@pytest.mark.parametrize("N", [1, 2, 3])
def test_product_is_as_accurate_as_fp32_multiply_adds(product, N, kind):
    """Right-hand sides at random, and those of smooth updates, whose product cancels by the condition of the
    matrix.  Root mean square over the cells of a Voronoi mesh of the relative L2 error: at P1, where
    the sums are short, both are within a few tenths of the representation's error, hence 1.1."""
    rng = np.random.default_rng(N)
    om = from_polymesh(periodic_voronoi(4 if N < 3 else 3), N)
    minvs, rs = [], []
    for cd in om.cells:
        m = np.linalg.inv(cd.M)
        r = rng.standard_normal((len(m), 5)) if kind == "random" else cd.M @ np.sin(3 * cd.nodes @ rng.standard_normal((3, 5)))
        minvs.append(0.5 * (m + m.T))
        rs.append(r.astype(np.float32))
    got = product(N, minvs, rs)
    err = {"pairs": [], "fp32": []}
    for m, r, y in zip(minvs, rs, got):
        exact = m @ r.astype(np.float64)
        err["pairs"].append(np.linalg.norm(y - exact) / np.linalg.norm(exact))
        err["fp32"].append(np.linalg.norm(_fp32(m, r) - exact) / np.linalg.norm(exact))
    pairs, fp32 = (float(np.sqrt(np.mean(np.square(err[k])))) for k in ("pairs", "fp32"))
    print(f"P{N} {kind}: pairs {pairs:.2e}, FP32 multiply-adds {fp32:.2e}")
    assert pairs <= 1.1 * fp32
