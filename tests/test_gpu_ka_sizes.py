"""Keyframe alignment evaluation at the edges of its launch shape: images of
one inner pixel, fewer pixels than a block, ragged rows, several pixels per
thread; with and without confidence; and a start no step improves (the
energy-only evaluations after three refused steps)."""
import numpy as np
import pytest

from oracle import ka

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def V():
    from paper_2104_06800_gb300 import voldor
    voldor.load()
    return voldor


def _pair(W, H, seed):
    rng = np.random.default_rng(seed)
    v, u = np.mgrid[0:H, 0:W].astype(np.float64)
    p = rng.uniform(0, 6, 4)
    Z = [4.0 + 0.02 * u + 0.03 * v + 0.05 * np.sin(u / 9 + p[2 * k]) + 0.05 * np.cos(v / 7 + p[2 * k + 1])
         for k in range(2)]
    for z in Z:
        z[rng.uniform(size=z.shape) < 0.03] = np.nan
    conf = rng.uniform(0.2, 1.0, size=(H, W)).astype(np.float32)
    K = (1.1 * W, 1.2 * W, W / 2.0 - 0.3, H / 2.0 + 0.2)
    T = np.array([[1, -0.004, 0.003, 0.02], [0.004, 1, -0.002, -0.01], [-0.003, 0.002, 1, 0.03]])
    return Z[0].astype(np.float32), Z[1].astype(np.float32), conf, K, T


@pytest.mark.parametrize("use_conf", [False, True])
@pytest.mark.parametrize("W,H", [(3, 3), (4, 5), (17, 9), (33, 31), (257, 3), (701, 467)])
def test_energy_and_count(V, W, H, use_conf):
    """float64 on both sides: the energies differ by the rounding of a sum of
    at most W H terms (1e-10 relative)."""
    import torch
    d1, d2, conf, K, T = _pair(W, H, W + H)
    dev = lambda x: torch.from_numpy(x).cuda()  # noqa: E731
    r = V.vd_ka_align(dev(d1), dev(d2), K, T, s0=1.01, conf2=dev(conf) if use_conf else None,
                      c=0.01, max_iters=0)
    n1, ok1 = ka.normals(d1, K)
    E, n = ka.energy(d1, n1, ok1, d2, conf if use_conf else None, K, T, 1.01, 0.01)
    assert r["n_valid"] == n and r["iterations"] == 0
    assert abs(r["energy"] - E) <= 1e-10 * abs(E)


def test_repeated_refusals_end_where_they_began(V):
    """Maps of independent noise: after the first steps none lowers E, lambda
    grows and the run ends; E is that of the returned estimate."""
    import torch
    d1, d2, conf, K, T = _pair(96, 64, 5)
    rng = np.random.default_rng(0)
    d2 = (d2 * (1 + 0.004 * rng.normal(size=d2.shape))).astype(np.float32)
    dev = lambda x: torch.from_numpy(x).cuda()  # noqa: E731
    r = V.vd_ka_align(dev(d1), dev(d2), K, T, s0=1.0, c=0.01, max_iters=50)
    again = V.vd_ka_align(dev(d1), dev(d2), K, r["T"], s0=r["s"], c=0.01, max_iters=0)
    assert r["iterations"] > 3
    assert again["energy"] == r["energy"] and again["n_valid"] == r["n_valid"]
    assert np.array_equal(again["cov"], r["cov"])
