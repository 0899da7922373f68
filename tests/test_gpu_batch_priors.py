"""A batch that gets new priors of the same kind runs its captured graph again,
on the new priors; a prior of another kind or baseline is another capture.  Each
run equals the window alone, bit for bit."""
import numpy as np
import pytest

from gpu_common import params_for, window
from test_gpu_batch import _results, _same

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def V():
    from paper_2104_06800_gb300 import voldor
    voldor.load()
    return voldor


def test_new_priors_replay_the_capture(V):
    w = window("rgbd_batch", 5300, size=(320, 240), N=3)
    p = V.vd_params_default(**params_for(w))
    desc = (w.W, w.H, w.N, w.intrinsics)
    other = (np.roll(w.depth_prior, 7, axis=1) * np.float32(1.02)).astype(np.float32)
    disp = (np.float32(0.3 * w.intrinsics[0]) / w.depth_prior).astype(np.float32)
    steps = [(lambda c: V.vd_push_depth_prior(c, w.depth_prior), 1),
             (lambda c: V.vd_push_depth_prior(c, other), 1),
             (lambda c: V.vd_push_stereo_prior(c, disp, 0.3), 2),
             (lambda c: V.vd_push_stereo_prior(c, disp, 0.25), 3),
             (lambda c: (V.vd_clear_prior(c), V.vd_push_depth_prior(c, other)), 4)]
    b = V.vd_batch_create([desc], [p])
    alone = V.vd_create(*desc, p)
    try:
        for push, captures in steps:
            for c in (V.vd_batch_window(b, 0), alone):
                for t in range(1, w.N + 1):
                    V.vd_push_flow(c, t, w.flow[t - 1])
                push(c)
            V.vd_batch_run(b, 2, V.VD_BATCH_BOOTSTRAP, 1)
            V.vd_bootstrap(alone)
            V.vd_run_em(alone, 2)
            assert _same(_results(V, V.vd_batch_window(b, 0), w), _results(V, alone, w)), captures
            assert V.vd_batch_get_stats(b)["captures"] == captures
    finally:
        V.vd_batch_destroy(b)
        V.vd_destroy(alone)
