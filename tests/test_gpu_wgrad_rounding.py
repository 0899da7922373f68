"""Rounding of the weight gradient's sums.  With a zero last layer its output is
0, the rigidness heads 1/2, and with targets of 0 every dL/dz of theirs is the
same power of two: the last layer's gradient is that times a sum of the layer's
own input, which float64 gives exactly enough."""
import numpy as np
import pytest

from test_gpu_cnn import RHO_MAX, RHO_MIN, _geom, _unpack

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def V():
    from paper_2104_06800_gb300 import voldor
    voldor.load()
    return voldor


def test_sums_of_one_sign(V):
    """The tensor core truncates its float32 sum once per MMA: of a chain of c
    MMAs with terms of one sign at most 2^-23 (c + 1) / 2 is lost, 3.0e-7 with
    the chains of 4 that are added in registers (with rounding to nearest, below
    that); a whole tile's 32 in one chain lose up to 2.0e-6 (3.6e-7 measured)."""
    import torch
    N, H, W = 4, 256, 512
    net = V.vd_cnn_create(N, seed=3)
    try:
        lay = V.vd_cnn_layout(net)
        theta = V.vd_cnn_get_params(net)
        theta[lay["w_offset"][5]:] = 0
        V.vd_cnn_set_params(net, theta)
        rng = np.random.default_rng(0)
        dev = lambda a: torch.from_numpy(a).cuda()  # noqa: E731
        flow = (rng.normal(size=(N, H, W, 2)) * 20).astype(np.float32)
        zeros = np.zeros((N, H, W), np.float32)
        V.vd_cnn_train_step(net, dev(flow), dev(np.ones((H, W), np.float32)), dev(zeros),
                            dev(np.ones((H, W), np.uint8)), RHO_MIN, RHO_MAX, 1.0, 0.0,
                            update=False, geom=_geom(0))
        dW, db = _unpack(V.vd_cnn_get_grads(net), lay)[5]
        a5 = V.vd_cnn_get_activation(net, 5, W, H, 32).astype(np.float64)
        c = 0.5 / (N * H * W)
        assert np.array_equal(db[1:], np.full(N, c * H * W))
        pad = np.pad(a5, ((1, 1), (1, 1), (0, 0)))
        want = np.array([[pad[ky:ky + H, kx:kx + W].sum((0, 1)) for kx in range(3)]
                         for ky in range(3)]) * c
        assert np.count_nonzero(want) > want.size // 2
        for co in range(1, 1 + N):
            assert np.linalg.norm(dW[co] - want) <= 3.0e-7 * np.linalg.norm(want)
    finally:
        V.vd_cnn_destroy(net)
