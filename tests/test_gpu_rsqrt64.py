"""The FP64 form's reciprocal square root over all exponents (both parities), the ends of the
mantissa range, the bits that its FP32 start cuts off, and the border to the subnormals,
against 80 or 128 bits: 0.501 ulp by its derivation, and rsqrt()'s 1 ulp for subnormals."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_0910_0121_gb300 import build as _build  # noqa: E402

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def rsqrt64():
    os.makedirs(_build.OBJ, exist_ok=True)
    lib = os.path.join(_build.OBJ, "rsqrt64_probe.so")
    subprocess.run([_build.nvcc(), "-shared", "-O3", "-std=c++17", *_build.ARCH, "-Xcompiler", "-fPIC",
                    *_build.EXTRA["force.cu"], "-I", _build.CSRC, "-o", lib, os.path.join(HERE, "rsqrt64_probe.cu")],
                   check=True)
    f = ctypes.CDLL(lib).rsqrt64_probe
    f.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_longlong]

    def call(x):
        X = torch.from_numpy(x).cuda()
        Y = torch.empty_like(X)
        torch.cuda.synchronize()
        assert f(X.data_ptr(), Y.data_ptr(), len(x)) == 0
        return Y.cpu().numpy()
    return call


def _ulps(x, y):
    ref = 1 / np.sqrt(x.astype(np.longdouble))
    return np.abs((y.astype(np.longdouble) - ref) / np.spacing(ref.astype(np.float64)).astype(np.longdouble)).max()


def test_normal_numbers(rsqrt64):
    rng = np.random.default_rng(64)
    ends = np.array([0, 1, 2, (1 << 29) - 1, 1 << 29, (1 << 52) - 1, (1 << 52) - (1 << 29), 1 << 51], np.uint64)
    for mant in (ends, rng.integers(0, 1 << 52, 400).astype(np.uint64),
                 rng.integers(0, 1 << 23, 200).astype(np.uint64) << np.uint64(29) | np.uint64((1 << 29) - 1)):
        ex = np.arange(1, 2047, dtype=np.uint64) << np.uint64(52)
        x = (ex[:, None] | mant[None, :]).ravel().view(np.float64)
        assert _ulps(x, rsqrt64(x)) <= 0.501
    x = rng.uniform(1.0, 4.0, 1 << 20)
    assert _ulps(x, rsqrt64(x)) <= 0.501


def test_subnormal_numbers(rsqrt64):
    rng = np.random.default_rng(65)
    bits = np.concatenate([np.arange(1, 65), (1 << 52) - np.arange(1, 65), 1 << np.arange(52),
                           rng.integers(1, 1 << 52, 4096)]).astype(np.uint64)
    x = bits.view(np.float64)
    assert _ulps(x, rsqrt64(x)) <= 1.0
