"""Chain propagation at the edges of its launch shapes: chains of 2 to 1300
pixels (fewer than the block's threads, one pass, many passes), every
direction, values that run along whole chains."""
import numpy as np
import pytest

from gpu_common import make_ctx, noisy_state, push_state, tie_band, window
from oracle import depth as odepth
from oracle import model as omodel

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def V():
    from paper_2104_06800_gb300 import voldor
    voldor.load()
    return voldor


@pytest.mark.parametrize("direction", [0, 1, 2, 3])
@pytest.mark.parametrize("size", [(2, 5), (31, 2), (64, 65), (257, 9), (11, 643), (1300, 3)])
def test_every_step_is_the_definition(V, size, direction):
    """K = 1: rho* is the given map.  One pixel in twelve holds the true
    depth, the others a random one, on noise-free flow: a true value is
    carried along its surface until the next one or an edge."""
    win = window("boxes640_stereo", 11, size=size, N=2, noisy=False)
    ctx, P, p = make_ctx(V, win, prior="none", n_hyp=1)
    try:
        rng = np.random.default_rng(direction)
        S = noisy_state(win, P, rng, rel=0.0)
        bad = rng.uniform(size=S.rho.shape) > 1.0 / 12.0
        lo, hi = win.params["rho_min"], win.params["rho_max"]
        S.rho[bad] = rng.uniform(lo, hi, size=int(bad.sum())).astype(np.float32)
        push_state(V, ctx, S)
        V.vd_depth_mstep(ctx, 0, direction)
        rs, es, new = (np.zeros((P.H, P.W), np.float32) for _ in range(3))
        V.vd_get_depth_candidates(ctx, rs, es)
        V.vd_get_inv_depth(ctx, new)
        assert np.array_equal(rs, S.rho)
        iu, iv = omodel.pixel_grid(P)
        own = omodel.energy(P, S, iu, iv, rs, p)
        band = tie_band(P, own)
        cu, cv = odepth.chain_coords(P, direction)
        prev = new[cv[0], cu[0]]
        assert np.array_equal(prev, rs[cv[0], cu[0]])
        run = longest = np.zeros(cu.shape[1], int)
        for m in range(1, cu.shape[0]):
            u, v = cu[m], cv[m]
            g = new[v, u]
            assert np.all((g == rs[v, u]) | (g == prev))
            Ep = omodel.energy(P, S, u, v, prev, p)
            took, kept = (g == prev) & (g != rs[v, u]), (g == rs[v, u]) & (g != prev)
            assert np.all(Ep[took] < own[v, u][took] + band[v, u][took])
            assert np.all(Ep[kept] >= own[v, u][kept] - band[v, u][kept])
            run = np.where(took, run + 1, 0)
            longest = np.maximum(longest, run)
            prev = g
        if cu.shape[0] >= 64:
            assert longest.max() >= 8      # the case does follow long runs
    finally:
        V.vd_destroy(ctx)

