"""The FP32 face fluxes' viscous coefficient and eps, formed without FP64 arithmetic, against FP64 values
rounded to FP32: rounded once, that is within 0.501 of the last place (48-bit factors), and equal but where
the FP64 value lies that close to the middle of two FP32 values."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def constants(tmp_path_factory):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2605_00619_gb300 import afe, build
    afe.lib()
    out = str(tmp_path_factory.mktemp("face") / "libface_constants.so")
    subprocess.run([build._nvcc(), "-O2", "-std=c++17", "-shared", "-Xcompiler", "-fPIC", "--expt-relaxed-constexpr",
                    *build.ARCH, "-I" + build.CSRC, "-I" + build.INCLUDE, os.path.join(HERE, "face_constants.cu"),
                    "-o", out], check=True)
    fn = ctypes.CDLL(out).face_constants
    fn.argtypes = [ctypes.c_int64] + [ctypes.c_void_p] * 4

    def run(a, b):
        da, db = (torch.from_numpy(x).cuda() for x in (a, b))
        p = torch.empty(len(a), dtype=torch.float32, device="cuda")
        e = torch.empty(3, len(a), dtype=torch.float32, device="cuda")
        torch.cuda.synchronize()
        assert fn(len(a), da.data_ptr(), db.data_ptr(), p.data_ptr(), e.data_ptr()) == 0
        return p.cpu().numpy(), e.cpu().numpy()
    return run


def _check(got, exact):
    ulp = np.spacing(np.abs(exact.astype(np.float32))).astype(np.float64)
    assert (np.abs(got.astype(np.float64) - exact) / ulp).max() <= 0.501
    assert np.mean(got == exact.astype(np.float32)) >= 0.995


@pytest.mark.parametrize("low,high,factor", [(-1, 1, None), (-20, 20, None), (-70, -40, 4 / 3), (30, 55, 1.97)])
def test_rounded_once(constants, low, high, factor):
    rng = np.random.default_rng(low + 100)
    n = 200000
    a, b = (2.0 ** rng.uniform(low, high, n) for _ in range(2))
    b[::3] = a[::3] * (1 + 1e-3 * rng.standard_normal(len(a[::3])))  # neighbours of about one size
    if factor is not None:
        b[:] = factor
    a[:50] = 1.0 - 2.0 ** -np.arange(2, 52)  # up to the next power of two
    product, eps = constants(a, b)
    _check(product, a * b)
    for N in (1, 2, 3):
        _check(eps[N - 1], (2 * N + 1) / ((a + b) * np.sqrt(np.pi / 2)))


def test_zero_and_tiny_values(constants):
    """No viscosity gives none; values that FP32 rounds to zero or to less than 24 bits as a conversion does."""
    a = np.array([0.0, 1e-300, 1e-42, 1e-40, 3e-38])
    product, _ = constants(a, np.full(5, 4 / 3))
    np.testing.assert_allclose(product, (a * 4 / 3).astype(np.float32), rtol=1e-6, atol=3e-45)
