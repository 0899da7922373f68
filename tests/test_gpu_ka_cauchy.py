"""A Cauchy scale without effect: every weight is the pixel's confidence, so the
covariance is that of c = 1e150 (where (r / c)^2 is 0 in float64 as well), bit
for bit, up to c = inf.  The energy is not defined there (inf * 0), and no step
is taken."""
import numpy as np
import pytest

from test_gpu_ka_sizes import _pair

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def V():
    from paper_2104_06800_gb300 import voldor
    voldor.load()
    return voldor


@pytest.mark.parametrize("c", [1e170, 1e305, 1.7e308, np.inf])
def test_least_squares_limit(V, c):
    import torch
    d1, d2, conf, K, T = _pair(96, 64, 2)
    dev = lambda x: torch.from_numpy(x).cuda()  # noqa: E731
    run = lambda c, n: V.vd_ka_align(dev(d1), dev(d2), K, T, s0=1.01, conf2=dev(conf),  # noqa: E731
                                     c=c, max_iters=n)
    want = run(1e150, 0)
    assert np.isfinite(want["cov"]).all() and want["n_valid"] > 1000
    for n in (0, 5):
        got = run(c, n)
        assert got["n_valid"] == want["n_valid"]
        assert np.array_equal(got["T"], T) and got["s"] == 1.01
        assert np.array_equal(got["cov"], want["cov"])
