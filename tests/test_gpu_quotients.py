"""Quotients from shared reciprocals against the division, over the ranges of
depths, residuals and scales."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
N = 1 << 22


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    import torch  # noqa: F401  (the CUDA runtime)
    from paper_2104_06800_gb300.build import ARCH, CSRC, INCLUDE, nvcc_path
    out = str(tmp_path_factory.mktemp("q") / "libvd_quotients.so")
    subprocess.run([nvcc_path(), "-O3", "-std=c++17", "-Xcompiler", "-fPIC", "-shared", *ARCH,
                    "-I", INCLUDE, "-I", CSRC,
                    os.path.join(ROOT, "tests", "native", "vd_quotients.cu"), "-o", out,
                    "-cudart", "shared"], check=True, capture_output=True)
    return C.CDLL(out)


def _both(fn, a, b):
    import torch
    ta, tb = torch.from_numpy(a).cuda(), torch.from_numpy(b).cuda()
    out = torch.zeros_like(ta), torch.zeros_like(ta)
    ptr = lambda t: C.c_void_p(t.data_ptr())  # noqa: E731
    torch.cuda.synchronize()
    assert fn(ptr(ta), ptr(tb), len(a), ptr(out[0]), ptr(out[1])) == 0
    return out[0].cpu().numpy(), out[1].cpu().numpy()


def _values(rng, lo, hi, dtype):
    return (rng.uniform(1, 2, N) * 2.0 ** rng.uniform(lo, hi, N)).astype(dtype)


def test_float64(lib):
    """What is rounded last is within 2^-51 units in the last place of a / b, so
    of 2^22 quotients none is expected to differ."""
    rng = np.random.default_rng(0)
    a, b = _values(rng, -40, 40, np.float64), _values(rng, -40, 40, np.float64)
    a *= rng.choice([-1, 1], N)
    a[:1000] = 0
    b[1000:2000] = 2.0 ** rng.integers(-40, 40, 1000)
    a[2000:3000] = b[2000:3000] * rng.integers(1, 1000, 1000)   # whole quotients
    fast, div = _both(lib.q_div64, a, b)
    assert np.array_equal(fast, div) and np.array_equal(div, a / b)


def test_packed_float32(lib):
    """Within 2^-23 units of a / b before the last rounding: a share of at most
    2^-22 of the quotients may be the neighbour (2^-20 allowed)."""
    rng = np.random.default_rng(1)
    a, b = _values(rng, -20, 33, np.float32), _values(rng, -10, 10, np.float32)
    a[:1000] = 0
    fast, div = _both(lib.q_div2, a, b)
    d = np.abs(fast.view(np.int32).astype(np.int64) - div.view(np.int32))
    assert d.max() <= 1 and np.mean(d > 0) <= 2.0 ** -20
