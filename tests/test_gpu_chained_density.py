"""Whole windows with the residual density's other forms, stage by stage against
the oracle: a scale that grows with the flow (alpha1 > 0, beta = 2: the per-pixel
scale of the pose scoring, the general form of the depth sampling) and other
shapes (beta != 2: the general form of both), with and without a prior, one flow
and several.  The bounds are those of the chained tests."""
import pytest

import synth
from chained import crop_problem, replay
from gpu_common import params_for
from oracle import model as omodel
from test_gpu_chained import _factory

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def V():
    from paper_2104_06800_gb300 import voldor
    voldor.load()
    return voldor


@pytest.mark.parametrize("N,size,alpha1,beta", [(3, (160, 120), 0.03, 2.0),
                                                (2, (131, 77), 0.0, 2.5),
                                                (1, (131, 77), 0.05, 2.0)])
def test_monocular(V, N, size, alpha1, beta):
    win = synth.make_window("planes160", 4)
    flow, K, _ = crop_problem(win, *size)
    kw = params_for(win, n_hyp=24, fisk_alpha1=alpha1, fisk_beta=beta)
    rep = replay(V, _factory(V, *size, N, K, flow[:N], V.vd_params_default(**kw)),
                 omodel.Problem(*size, N, K, flow[:N]), omodel.Params(**kw), 2,
                 f"N {N} alpha1 {alpha1} beta {beta}")
    print(rep.summary())


@pytest.mark.parametrize("name,size,N,alpha1,beta", [
    ("boxes640_stereo", (160, 120), 4, 0.02, 1.5),
    ("rgbd_batch", (97, 83), 5, 0.01, 2.0),
])
def test_with_a_prior(V, name, size, N, alpha1, beta):
    win = synth.make_window(name, 4, size=size, N=N)
    kw = params_for(win, n_hyp=24, fisk_alpha1=alpha1, fisk_beta=beta)
    P = omodel.problem_from_window(win)
    stereo = (win.stereo_disp, win.stereo_baseline) if P.prior_kind == "stereo" else None
    rgbd = win.depth_prior if P.prior_kind == "rgbd" else None
    rep = replay(V, _factory(V, win.W, win.H, win.N, win.intrinsics, win.flow,
                             V.vd_params_default(**kw), stereo=stereo, depth_prior=rgbd),
                 P, omodel.Params(**kw), 2, f"{name} alpha1 {alpha1} beta {beta}")
    print(rep.summary())
