"""Chains up to the longest an image may have (16384 pixels): propagation with
more shared memory than a block has by default and with many pixels a thread,
smoothing without its staging (above 6112 pixels); and the parts of the
hierarchical propagation, coarse cells and restart windows of ragged sizes."""
import numpy as np
import pytest

import chained
from gpu_common import make_ctx, noisy_state, push_state, tie_band, window
from oracle import depth as odepth
from oracle import model as omodel
from test_gpu_propagate import test_every_step_is_the_definition as every_step

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def V():
    from paper_2104_06800_gb300 import voldor
    voldor.load()
    return voldor


@pytest.mark.parametrize("size,direction", [((6200, 2), 0), ((3, 4500), 3), ((4093, 5), 2),
                                            ((2, 16384), 1)])
def test_propagation(V, size, direction):
    every_step(V, size, direction)


@pytest.mark.parametrize("size,direction", [((6112, 3), 0), ((6200, 2), 2), ((3, 6113), 1)])
def test_smoothing(V, size, direction):
    win = window("boxes640_stereo", 12, size=size, N=2)
    ctx, P, p = make_ctx(V, win, prior="none")
    try:
        S = noisy_state(win, P, np.random.default_rng(4), rel=0.01)
        push_state(V, ctx, S)
        chained.estep_stage(V, ctx, P, S, direction, p, chained.Report("long"), "estep")
    finally:
        V.vd_destroy(ctx)


def _hier(V, size, direction, scale, restart, spoil):
    """One depth step with K = 1 (rho* is the given map: the true depth at one
    pixel in twelve, random elsewhere); (problem, state, rho*, result, E, band)."""
    win = window("boxes640_stereo", 13, size=size, N=2, noisy=False)
    ctx, P, p = make_ctx(V, win, prior="none", n_hyp=1, hierarchical=1, hier_scale=scale,
                         hier_window=restart)
    try:
        rng = np.random.default_rng(direction)
        S = noisy_state(win, P, rng, rel=0.0)
        bad = rng.uniform(size=S.rho.shape) > 1.0 / 12.0
        lo, hi = win.params["rho_min"], win.params["rho_max"]
        S.rho[bad] = rng.uniform(lo, hi, size=int(bad.sum())).astype(np.float32)
        if spoil:
            S.rho[0, 0] = hi
        push_state(V, ctx, S)
        V.vd_depth_mstep(ctx, 0, direction)
        rs, es, new = (np.zeros((P.H, P.W), np.float32) for _ in range(3))
        V.vd_get_depth_candidates(ctx, rs, es)
        V.vd_get_inv_depth(ctx, new)
    finally:
        V.vd_destroy(ctx)
    assert np.array_equal(rs, S.rho)
    iu, iv = omodel.pixel_grid(P)
    own = omodel.energy(P, S, iu, iv, rs, p)
    return P, S, p, rs, new, own, tie_band(P, own)


def _check(P, S, p, u, v, offered, g, rs, own, band):
    """g at pixels (u, v) is `offered` where its energy is below rho*'s, else rho*."""
    mine = rs[v, u]
    assert np.all((g == mine) | (g == offered))
    E = omodel.energy(P, S, u, v, offered, p)
    took, kept = (g == offered) & (g != mine), (g == mine) & (g != offered)
    assert np.all(E[took] < own[v, u][took] + band[v, u][took])
    assert np.all(E[kept] >= own[v, u][kept] - band[v, u][kept])
    return int(took.sum())


@pytest.mark.parametrize("direction", [0, 1, 2, 3])
@pytest.mark.parametrize("size,scale", [((97, 41), 1), ((97, 41), 3), ((64, 50), 7), ((41, 700), 5)])
def test_coarse_pass(V, size, scale, direction):
    """A window of one pixel leaves what the coarse pass gave.  A cell's value
    is that of its representative pixel, which is offered its own."""
    P, S, p, rs, new, own, band = _hier(V, size, direction, scale, 1, False)
    ru = np.minimum(np.arange((P.W + scale - 1) // scale) * scale, P.W - 1)
    rv = np.minimum(np.arange((P.H + scale - 1) // scale) * scale, P.H - 1)
    cu, cv = np.meshgrid(ru, rv)
    coarse = new[cv, cu]
    along = (lambda a: a) if direction in (0, 2) else np.transpose
    order = slice(None) if direction < 2 else slice(None, None, -1)
    c, u, v = (along(a)[:, order] for a in (coarse, cu, cv))
    assert np.array_equal(c[:, 0], rs[v[:, 0], u[:, 0]])
    taken = sum(_check(P, S, p, u[:, m], v[:, m], c[:, m - 1], c[:, m], rs, own, band)
                for m in range(1, c.shape[1]))
    assert taken > 0
    iu, iv = omodel.pixel_grid(P)
    taken = _check(P, S, p, iu, iv, coarse[iv // scale, iu // scale], new, rs, own, band)
    assert taken > 0


@pytest.mark.parametrize("direction", [0, 1, 2, 3])
@pytest.mark.parametrize("size,restart", [((97, 41), 5), ((33, 64), 16), ((300, 7), 64),
                                          ((70, 30), 2000)])
def test_restart_windows(V, size, restart, direction):
    """A cell larger than the image offers every pixel the value of pixel
    (0, 0), which is spoiled: what moves is the windows' walk."""
    P, S, p, rs, new, own, band = _hier(V, size, direction, 5000, restart, True)
    iu, iv = omodel.pixel_grid(P)
    E_spoiled = omodel.energy(P, S, iu, iv, np.full_like(rs, rs[0, 0]), p)
    calm = (E_spoiled > own + band) | (rs == rs[0, 0])   # not offered anything better by the cell
    cu, cv = odepth.chain_coords(P, direction)
    taken = 0
    for m in range(cu.shape[0]):
        u, v = cu[m], cv[m]
        k = calm[v, u]
        g = new[v, u]
        if m % restart == 0:
            assert np.array_equal(g[k], rs[v, u][k])
        else:
            taken += _check(P, S, p, u[k], v[k], new[cv[m - 1], cu[m - 1]][k], g[k], rs, own, band)
    assert calm.mean() > 0.5 and taken > 0
