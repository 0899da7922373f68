"""The scratch that the standalone calls keep between calls: bounded, given back
to whatever else of the library needs memory."""
import fake_cuda

ALIGN = """
class KA(C.Structure):
    _fields_ = [("pose", C.c_double * 12), ("s", C.c_double), ("cauchy_c", C.c_double),
                ("fix_scale", C.c_int), ("max_iters", C.c_int), ("cov", C.c_double * 36),
                ("energy", C.c_double), ("iterations", C.c_int), ("n_valid", C.c_longlong)]


def align(W=320, H=240):
    a, b = dev(4 * W * H), dev(4 * W * H)
    io = KA(s=1.0, cauchy_c=0.01, max_iters=3)
    for i in (0, 5, 10):
        io.pose[i] = 1.0
    K = (C.c_double * 4)(300.0, 300.0, W / 2, H / 2)
    ok(lib.vd_ka_align(a, b, None, W, H, K, C.byref(io), None))
    assert fake.cudaFree(a) == 0 and fake.cudaFree(b) == 0


def score(n=100, m=256):
    pts, obs, poses, out, K = dev(16 * n), dev(16 * n), dev(96 * m), dev(8 * m), dev(32)
    ok(lib.vd_score_poses(pts, obs, n, poses, m, K, F(2.0), F(1e-3), out, None))
    for p in (pts, obs, poses, out, K):
        assert fake.cudaFree(p) == 0
"""


def test_the_pool_is_bounded():
    fake_cuda.run(ALIGN + """
align(2000, 1500)                             # 96 MB of normals
assert 0 < fake.fake_idle(0) <= 32 << 20
assert fake.fake_used(0) == 0
""")


def test_a_network_finds_the_pools_memory():
    """Room for a network and its images, but not for the idle scratch beside."""
    fake_cuda.run(ALIGN + """
def train(W=160, H=120, N=6):
    net = P()
    ok(lib.vd_cnn_create(N, C.c_ulonglong(0), C.byref(net)))
    flow = dev(8 * W * H * N)
    ok(lib.vd_cnn_forward(net, flow, W, H, None, F(0.1), F(2.0), None, None, None))
    used = fake.fake_used(0)
    ok(lib.vd_cnn_destroy(net))
    assert fake.cudaFree(flow) == 0
    return used


def create_only():
    net = P()
    ok(lib.vd_cnn_create(6, C.c_ulonglong(0), C.byref(net)))
    used = fake.fake_used(0)
    ok(lib.vd_cnn_destroy(net))
    return used


for need in (create_only, train):
    room = need()
    align()
    assert fake.fake_idle(0) > 0
    fake.fake_capacity(room + fake.fake_idle(0) // 2)
    need()
    assert fake.fake_idle(0) == 0
    fake.fake_capacity(64 << 30)
""")


def test_scratch_beyond_the_kept_finds_room():
    fake_cuda.run(ALIGN + """
align()
kept = fake.fake_idle(0)
fake.fake_capacity(64 << 20)
align(1200, 700)                              # 27 MB of normals and the images
score()
""")


def test_scratch_without_memory_is_an_error_that_leaves_none_behind():
    fake_cuda.run(ALIGN + """
n, m = 100, 1024
pts, obs, poses, out, K = dev(16 * n), dev(16 * n), dev(96 * m), dev(8 * m), dev(32)
fake.fake_capacity(fake.fake_used(0) + 1000)
assert lib.vd_score_poses(pts, obs, n, poses, m, K, F(2.0), F(1e-3), out, None) == -3
assert fake.cudaGetLastError() == 0
""")


def test_calls_after_a_device_reset():
    """A reset ends the pool with its context; neither call may use it again."""
    fake_cuda.run(ALIGN + """
for call in (score, align):
    call()
    assert fake.cudaDeviceReset() == 0
    call()
    assert fake.fake_dead_pool_uses() == 0
# the allocations that would trim the dead pool
assert fake.cudaDeviceReset() == 0
fake.fake_capacity(1000)
net = P()
assert lib.vd_cnn_create(6, C.c_ulonglong(0), C.byref(net)) == -3
assert fake.fake_dead_pool_uses() == 0
""")


def test_one_pool_per_device():
    fake_cuda.run(ALIGN + """
for d in (0, 1, 0, 1, 0):
    assert fake.cudaSetDevice(d) == 0
    align()
    score()
assert fake.fake_pools() == 2 and fake.fake_dead_pool_uses() == 0
for d in (0, 1):
    assert 0 < fake.fake_idle(d) <= 32 << 20 and fake.fake_used(d) == 0
""")
