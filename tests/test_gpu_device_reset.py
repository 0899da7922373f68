"""The standalone calls in a process that resets its device between them (a
child process: a reset ends everything the process has on the device)."""
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

CODE = """
import ctypes as C
import numpy as np
import torch                       # loads the CUDA runtime; not used otherwise
from paper_2104_06800_gb300 import build, voldor as V

build.build()
lib = V.load()
rt = C.CDLL("libcudart.so.13")


def dev(a):
    p = C.c_void_p()
    assert rt.cudaMalloc(C.byref(p), C.c_size_t(a.nbytes)) == 0
    assert rt.cudaMemcpy(p, a.ctypes.data_as(C.c_void_p), C.c_size_t(a.nbytes), 1) == 0
    return p


def score(n=3000, m=40):
    rng = np.random.default_rng(0)
    X = rng.uniform(-1, 1, (n, 4)).astype(np.float32)
    X[:, 2] += 5
    X[:, 3] = 1
    obs = rng.uniform(50, 250, (n, 4)).astype(np.float32)
    obs[:, 2] = 0.8
    poses = np.tile(np.eye(3, 4).reshape(1, 12), (m, 1))
    poses[:, 3] = rng.normal(size=m) * 0.1
    e = np.zeros(m)
    out = dev(e)
    assert lib.vd_score_poses(dev(X), dev(obs), n, dev(poses), m,
                              dev(np.array([300.0, 300.0, 160.0, 120.0])), 2.0, 1e-3, out,
                              None) == 0, lib.vd_last_error()
    assert rt.cudaMemcpy(e.ctypes.data_as(C.c_void_p), out, C.c_size_t(e.nbytes), 2) == 0
    return e


def align(W=120, H=90):
    v, u = np.mgrid[0:H, 0:W]
    Z = (4 + 0.01 * u + 0.02 * v + 0.1 * np.sin(u / 7)).astype(np.float32)
    io = V.vd_ka(s=1.01, cauchy_c=0.01, max_iters=4)
    for i in (0, 5, 10):
        io.pose[i] = 1.0
    k = (C.c_double * 4)(130.0, 130.0, W / 2, H / 2)
    assert lib.vd_ka_align(dev(Z), dev(Z), None, W, H, k, C.byref(io), None) == 0
    return np.array(io.pose[:] + [io.s, io.energy])


first = score(), align()
assert np.isfinite(first[0]).all() and np.isfinite(first[1]).all()
for _ in range(2):
    assert rt.cudaDeviceReset() == 0
    assert np.array_equal(score(), first[0]) and np.array_equal(align(), first[1])
print("same")
"""


def test_scoring_and_alignment_after_a_reset():
    r = subprocess.run([sys.executable, "-c", CODE], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.endswith("same\n"), r.stdout + r.stderr[-3000:]
