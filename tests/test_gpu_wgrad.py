"""Weight gradient at the edges of its tiles: images of one pixel, of one
16-pixel step, one pixel more or less than a 128-pixel tile or a 4-row block,
and several tiles with ragged last ones; 16 and 32 input planes."""
import numpy as np
import pytest

from oracle import cnn
from test_gpu_cnn import RHO_MAX, RHO_MIN, W_Q, _acts, _geom, _setup, _unpack

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def V():
    from paper_2104_06800_gb300 import voldor
    voldor.load()
    return voldor


@pytest.mark.parametrize("N,H,W", [(2, 1, 1), (2, 3, 16), (8, 5, 17), (2, 4, 127), (8, 9, 128),
                                   (2, 6, 129), (8, 13, 272)])
def test_gradients_at_tile_edges(V, N, H, W):
    """Both sides store dL/dz of every layer in bf16; one that rounds the other
    way differs by 2^-8 of itself, and layer l's has passed 6 - l such
    roundings: a normwise bound of (6 - l) 2^-8, where a tap, row or pixel
    left out or counted twice is of the order of its share of the sum."""
    net, lay, theta, flow, rho_t, q_t, mask, T = _setup(V, N, H, W, seed=5)
    mask[:] = 1
    try:
        V.vd_cnn_train_step(net, T(flow), T(rho_t), T(q_t), T(mask), RHO_MIN, RHO_MAX, W_Q, 0.0,
                            update=False, geom=_geom(5))
        a, z = _acts(V, net, lay, W, H)
        _, dz = cnn.loss_and_grad(z, rho_t.astype(np.float64), q_t.astype(np.float64), mask,
                                  RHO_MIN, RHO_MAX, W_Q)
        grads = cnn.backward(_unpack(theta, lay), a, [a[l + 1] for l in range(5)] + [z], dz)
        got = _unpack(V.vd_cnn_get_grads(net), lay)
        for l in range(6):
            for g, ref in zip(got[l], grads[l]):
                assert np.linalg.norm(g - ref) <= (6 - l) * 2.0 ** -8 * np.linalg.norm(ref) + 1e-12, l
    finally:
        V.vd_cnn_destroy(net)
