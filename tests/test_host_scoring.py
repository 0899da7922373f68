"""Host code of the standalone scoring: where its intrinsics may come from."""
import pytest

import fake_cuda

SCORE = """
import struct
K = (720.0, 710.0, 608.5, 184.25)


def score(name, intrinsics, stream=None, n=100, m=7):
    pts, obs, poses, out = dev(16 * n), dev(16 * n), dev(96 * m), dev(8 * m)
    s = getattr(lib, name)(pts, obs, n, poses, m, intrinsics, F(2.0), F(1e-3), out, stream)
    for p in (pts, obs, poses, out):
        assert fake.cudaFree(p) == 0
    return s


def read():
    k = (C.c_double * 4)()
    how = fake.fake_intrinsics(k)
    assert how >= 0, "read at a misaligned address"
    return how, tuple(k)


def device_copy(offset):
    p = dev(64)
    C.memmove(p.value + offset, struct.pack("4d", *K), 32)
    return P(p.value + offset)
"""


@pytest.mark.parametrize("name", ["vd_score_poses", "vd_score_poses_noalloc"])
@pytest.mark.parametrize("offset", [0, 4, 8, 1])
def test_device_intrinsics_of_any_alignment(name, offset):
    """They were fetched by a copy, which takes any address; a kernel that reads
    them as float64 needs one of 8 bytes."""
    fake_cuda.run(SCORE + f"""
ok(score({name!r}, device_copy({offset})))
how, k = read()
assert how == 0 or k == K
""")


@pytest.mark.parametrize("name", ["vd_score_poses", "vd_score_poses_noalloc"])
def test_other_streams_wait_for_the_default_stream(name):
    """On a stream of the caller's that does not wait for the default stream,
    the copy has to: it blocks, as it always did."""
    fake_cuda.run(SCORE + f"""
before = fake.fake_blocking_copies()
ok(score({name!r}, device_copy(0), stream=P(0x1000)))
assert fake.fake_blocking_copies() == before + 1
""")


@pytest.mark.parametrize("name", ["vd_score_poses", "vd_score_poses_noalloc"])
def test_host_intrinsics(name):
    fake_cuda.run(SCORE + f"""
host = (C.c_double * 4)(*K)
for stream in (None, P(0x1000)):
    ok(score({name!r}, C.cast(host, P), stream))
    assert read()[0] == 0                     # they travel as kernel arguments
""")
