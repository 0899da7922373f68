"""The network's kernels on a second device of the process: their shared memory
has to be granted, and their grids sized, on each device a network lives on."""
import fake_cuda

STEP = """
def step(n_flows, W, H):
    net = P()
    ok(lib.vd_cnn_create(n_flows, C.c_ulonglong(0), C.byref(net)))
    flow, rho, q = dev(8 * W * H * n_flows), dev(4 * W * H), dev(4 * W * H * n_flows)
    mask, loss = dev(W * H), C.c_double()
    ok(lib.vd_cnn_train_step(net, flow, W, H, None, rho, q, mask, F(0.1), F(2.0), F(1.0), F(1e-3),
                             0, C.byref(loss), None))
    ok(lib.vd_cnn_forward(net, flow, W, H, None, F(0.1), F(2.0), rho, q, None))
    ok(lib.vd_cnn_destroy(net))
"""


def test_training_on_a_second_device():
    """6 flows take 16 input planes, 8 take 32: every instantiation launches."""
    fake_cuda.run(STEP + """
for d in (0, 1, 0):
    assert fake.cudaSetDevice(d) == 0
    for n in (6, 8):
        step(n, 640, 480)
""")


def test_grids_follow_the_device():
    """640 x 480 is more tiles than either device has SMs (152 and 20 in the
    fake, one resident block each)."""
    fake_cuda.run(STEP + """
assert fake.cudaSetDevice(1) == 0
step(6, 640, 480)
assert fake.fake_max_persistent_grid() == 20
assert fake.cudaSetDevice(0) == 0
step(6, 640, 480)
assert fake.fake_max_persistent_grid() == 152
""")


def test_training_after_a_device_reset():
    fake_cuda.run(STEP + """
step(6, 64, 48)
assert fake.cudaDeviceReset() == 0
step(6, 64, 48)
""")
