"""A residual of exactly zero under the general form of the density (a scale per
point or per flow vector): with beta = 2 the density at the origin is finite,
beta / (2 pi alpha^2), and so are the energies and posteriors."""
import numpy as np
import pytest

from gpu_common import RIGID_TOL, push_state, tie_band
from oracle import hmm
from oracle import model as omodel
from oracle import pose as opose

pytestmark = pytest.mark.gpu

P0 = 1e-3


@pytest.fixture(scope="module")
def V():
    from paper_2104_06800_gb300 import voldor
    voldor.load()
    return voldor


@pytest.mark.parametrize("beta", [1.5, 2.0, 2.5])
@pytest.mark.parametrize("name", ["vd_score_poses", "vd_score_poses_noalloc"])
def test_scoring(V, name, beta):
    """Points on the optical axis at depth 1 are seen at (cx, cy) exactly."""
    import torch
    K = (300.0, 310.0, 160.0, 120.0)
    n = 70
    rng = np.random.default_rng(0)
    pts = np.tile(np.array([0, 0, 1, 1], np.float32), (n, 1))
    pts[:, 3] = rng.uniform(0.2, 1, n)
    obs = np.tile(np.array([K[2], K[3], 0, 0], np.float32), (n, 1))
    obs[:, 2] = rng.uniform(0.4, 1.2, n)
    obs[::3, 0] += 1.5                         # others beside them
    dev = lambda a: torch.from_numpy(a).cuda()  # noqa: E731
    e = torch.zeros(2, dtype=torch.float64, device="cuda")
    poses = np.tile(np.eye(3, 4).reshape(1, 12), (2, 1))
    getattr(V, name)(dev(pts), dev(obs), dev(poses), dev(np.array(K)), beta, P0, e)
    P = omodel.Problem(10, 10, 1, K, np.zeros((1, 10, 10, 2), np.float32))
    rs = dict(X=pts[:, :3].astype(np.float64), xobs=obs[:, :2].astype(np.float64),
              w=pts[:, 3].astype(np.float64), alpha=obs[:, 2].astype(np.float64))
    want = opose.score(P, np.eye(3, 4), rs, omodel.Params(fisk_beta=beta, outlier_density=P0))
    assert np.allclose(e.cpu().numpy(), want, rtol=1e-4)


@pytest.mark.parametrize("N", [1, 3])
def test_window(V, N):
    """No motion, no flow, an intrinsic matrix of powers of two: every residual
    is zero in float32 as well."""
    W, H, K = 64, 32, (64.0, 64.0, 32.0, 16.0)
    flow = np.zeros((N, H, W, 2), np.float32)
    par = dict(fisk_alpha0=0.5, fisk_alpha1=0.02, rho_min=0.25, rho_max=4.0, n_hyp=8)
    ctx = V.vd_create(W, H, N, K, V.vd_params_default(**par))
    try:
        P, p = omodel.Problem(W, H, N, K, flow), omodel.Params(**par)
        rng = np.random.default_rng(1)
        S = omodel.State(rho=rng.uniform(0.5, 2, (H, W)).astype(np.float32),
                         q=rng.uniform(0.2, 1, (N, H, W)).astype(np.float32),
                         qhat=np.ones((H, W), np.float32),
                         G=np.tile(np.eye(3, 4), (N + 1, 1, 1)))
        for t in range(1, N + 1):
            V.vd_push_flow(ctx, t, flow[t - 1])
        push_state(V, ctx, S)
        e = np.zeros((H, W), np.float32)
        V.vd_eval_energy(ctx, S.rho, e)
        iu, iv = omodel.pixel_grid(P)
        want = omodel.energy(P, S, iu, iv, S.rho, p)
        assert np.all(np.abs(e - want) <= tie_band(P, want))
        V.vd_depth_mstep(ctx, 0, 0)
        V.vd_get_depth_candidates(ctx, np.zeros((H, W), np.float32), e)
        assert np.all(np.isfinite(e)) and np.all(np.abs(e - want) <= tie_band(P, want))
        push_state(V, ctx, S)
        V.vd_rigidness_estep(ctx, 0)
        q = np.zeros((N, H, W), np.float32)
        V.vd_get_rigidness(ctx, q)
        ref, _, _ = hmm.rigidness_estep(P, S, S.rho, 0, p)
        assert np.max(np.abs(q - ref)) <= RIGID_TOL
    finally:
        V.vd_destroy(ctx)
