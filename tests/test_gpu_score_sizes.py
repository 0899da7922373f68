"""Dense pose scoring at the edges of its passes: pixel counts around a pair of
32-pixel rows, a pass of 128 and a block; pose counts around the groups of 8 and
32; points behind the camera, weights of zero and residuals whose likelihood
ratio overflows float32; beta = 2 (a scale per point) and another beta."""
import numpy as np
import pytest

from oracle import geometry as ogeo
from oracle import model as omodel
from oracle import pose as opose

pytestmark = pytest.mark.gpu

K = (300.0, 310.0, 160.0, 120.0)
# Image positions are below 500 px in float32: four roundings of 2^-24 * 500 px
# each displace a residual r by at most d = 1.2e-4 px, and a term's relative
# error is at most |d log y / dr| d = 4 r d / (alpha^2 + r^2) <= 2 d / alpha =
# 6e-4 for alpha >= 0.4.
RTOL = 1e-3


@pytest.fixture(scope="module")
def V():
    from paper_2104_06800_gb300 import voldor
    voldor.load()
    return voldor


@pytest.mark.parametrize("beta", [2.0, 2.5])
@pytest.mark.parametrize("n,m", [(1, 1), (31, 7), (33, 8), (63, 9), (65, 31), (127, 32), (129, 33),
                                 (1025, 65), (39001, 3)])
def test_score_sizes(V, n, m, beta):
    import torch
    rng = np.random.default_rng(n * 100 + m)
    X = rng.uniform(-0.4, 0.4, size=(n, 3))
    X[:, 2] = rng.uniform(2, 20, size=n)
    X[:, :2] *= X[:, 2:]
    w = np.where(rng.uniform(size=n) < 0.1, 0.0, rng.uniform(0.2, 1, size=n))
    poses = np.stack([ogeo.se3_exp(rng.normal(size=6) * 0.02) for _ in range(m)])
    xobs = np.stack([K[0] * X[:, 0] / X[:, 2] + K[2], K[1] * X[:, 1] / X[:, 2] + K[3]], 1)
    xobs += rng.normal(size=xobs.shape)
    alpha = rng.uniform(0.4, 1.2, size=n)
    if n > 32:
        xobs[5] += 3e9          # log(1 + y) with y beyond float32
        X[7, 2] = -3.0          # behind every camera
    pts = np.concatenate([X, w[:, None]], 1).astype(np.float32)
    obs = np.concatenate([xobs, alpha[:, None], np.zeros((n, 1))], 1).astype(np.float32)
    e = torch.zeros(m, dtype=torch.float64, device="cuda")
    V.vd_score_poses(torch.from_numpy(pts).cuda(), torch.from_numpy(obs).cuda(),
                     torch.from_numpy(poses.reshape(m, 12)).cuda(),
                     torch.tensor(K, dtype=torch.float64, device="cuda"), beta, 1e-3, e)
    P = omodel.Problem(10, 10, 1, K, np.zeros((1, 10, 10, 2), np.float32))
    p = omodel.Params(fisk_beta=beta, outlier_density=1e-3)
    rs = dict(X=pts[:, :3].astype(np.float64), xobs=obs[:, :2].astype(np.float64),
              w=pts[:, 3].astype(np.float64), alpha=obs[:, 2].astype(np.float64))
    want = np.array([opose.score(P, G, rs, p) for G in poses])
    assert np.allclose(e.cpu().numpy(), want, rtol=RTOL, atol=1e-12)
