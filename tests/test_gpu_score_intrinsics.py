"""Intrinsics of the standalone scoring: the same energies from device memory of
any alignment, from host memory, and from device memory that the default stream
fills while the call runs on a stream of its own."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

K = (300.0, 310.0, 160.0, 120.0)


@pytest.fixture(scope="module")
def V():
    from paper_2104_06800_gb300 import voldor
    voldor.load()
    return voldor


class _At:
    def __init__(self, tensor, offset):
        self.tensor, self.offset = tensor, offset

    def data_ptr(self):
        return self.tensor.data_ptr() + self.offset


def _scene(n=5000, m=9):
    import torch
    rng = np.random.default_rng(3)
    X = np.concatenate([rng.uniform(-2, 2, (n, 2)), rng.uniform(2, 9, (n, 1)),
                        rng.uniform(0.1, 1, (n, 1))], 1)
    obs = np.stack([K[0] * X[:, 0] / X[:, 2] + K[2], K[1] * X[:, 1] / X[:, 2] + K[3],
                    np.full(n, 0.7), np.zeros(n)], 1)
    obs[:, :2] += rng.normal(size=(n, 2))
    poses = np.tile(np.eye(3, 4).reshape(1, 12), (m, 1))
    poses[:, [3, 7, 11]] += 0.01 * rng.normal(size=(m, 3))
    dev = lambda a, t: torch.from_numpy(a.astype(t)).cuda()  # noqa: E731
    return dev(X, np.float32), dev(obs, np.float32), dev(poses, np.float64)


@pytest.mark.parametrize("name", ["vd_score_poses", "vd_score_poses_noalloc"])
def test_where_intrinsics_may_come_from(V, name):
    import torch
    pts, obs, poses = _scene()
    k = torch.tensor(K, dtype=torch.float64)
    score = getattr(V, name)
    out = lambda: torch.full((len(poses),), -1.0, dtype=torch.float64, device="cuda")  # noqa: E731
    side = torch.cuda.Stream()
    want = score(pts, obs, poses, k.cuda(), 2.0, 1e-3, out()).cpu()
    assert torch.isfinite(want).all() and len(set(want.tolist())) > 1
    raw = torch.zeros(64, dtype=torch.uint8, device="cuda")
    for offset in (4, 8, 13):
        raw[offset:offset + 32] = k.cuda().view(torch.uint8)
        torch.cuda.synchronize()
        for stream in (None, side.cuda_stream):
            got = score(pts, obs, poses, _At(raw, offset), 2.0, 1e-3, out(), stream=stream)
            assert torch.equal(got.cpu(), want), (offset, stream)
    for stream in (None, side.cuda_stream):
        assert torch.equal(score(pts, obs, poses, k, 2.0, 1e-3, out(), stream=stream).cpu(), want)
    # the default stream writes them some 20 ms after the call began
    late, e = torch.tensor([1.0, 1.0, 0.0, 0.0], dtype=torch.float64, device="cuda"), out()
    right = k.cuda()
    torch.cuda.synchronize()
    torch.cuda._sleep(40_000_000)
    late.copy_(right)
    assert torch.equal(score(pts, obs, poses, late, 2.0, 1e-3, e, stream=side.cuda_stream).cpu(),
                       want)
