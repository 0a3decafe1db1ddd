"""The placement by a cluster of eight blocks (more axis pixels than one block holds) against the oracle,
decision for decision: candidates in shared and in global memory, elements ranked and not, and problems
of both forms in one handle."""
import numpy as np
import pytest

from paper_2406_04008_gb300 import workloads as W
from tests.test_gpu_mat import _check, env  # noqa: F401  (the fixture)

pytestmark = pytest.mark.gpu


def _problem(rings, n, grid, seed=3):
    rng = W.PCG32(seed)
    els, params = [], []
    for _ in range(n):
        els.append((1, W.regular_polygon(0.002 + 0.02 * rng.uniform() ** 2, 7), 0.0))
        params.append((0.5, 0.5, 6.0 * rng.uniform(), 0.6 + 0.8 * rng.uniform()))
    return W.make_problem(els, rings, params, grid)


def _star():
    a = 0.32 + 2.0 * np.pi * np.arange(24) / 24
    r = np.where(np.arange(24) % 2 == 0, 0.47, 0.25)
    return [0.5 + np.stack([r * np.cos(a), r * np.sin(a)], 1)]


def _comb(grid):
    # strips two pixels wide with one between them: every inside pixel is on the axis
    x = np.arange(1, grid - 2, 3) / grid
    return [np.array([(u, 0.01), (u + 2 / grid, 0.01), (u + 2 / grid, 0.99), (u, 0.99)]) for u in x]


def _greedy(prob, axis, width, grid):
    """The placement's rule (elements by decreasing radius, then index; each at the widest axis pixel with room,
    else the one of largest clearance; the lower pixel on a tie) on given maps, in float32."""
    f = np.float32
    pix = np.flatnonzero(axis)
    x, y, w = pix % grid, pix // grid, np.rint(width[pix].astype(np.float64) ** 2).astype(np.int64)
    pts, off, q = prob["pts"].reshape(-1, 2), prob["pt_off"], prob["params0"].reshape(-1, 4).copy()
    rbin = np.array([np.sqrt((pts[a:b].astype(np.float64) ** 2).sum(1)).max() for a, b in zip(off, off[1:])], f)
    r = rbin * q[:, 3] * f(grid)
    clear = np.full(len(pix), np.finfo(f).max, f)
    for e in np.argsort(-r, kind="stable"):
        room = np.flatnonzero(clear >= r[e])
        k = room[np.argmax(w[room])] if len(room) else np.argmax(clear)
        q[e, :2] = (f(x[k]) + f(0.5)) / f(grid), (f(y[k]) + f(0.5)) / f(grid)
        d2 = ((x - x[k]) ** 2 + (y - y[k]) ** 2).astype(f)
        clear = np.minimum(clear, np.sqrt(d2) - r[e])
    return q


@pytest.mark.parametrize("n", [1, 70])
def test_star_beyond_one_block(env, n):
    # 21 k axis pixels
    _check(env, [_problem(_star(), n, 1352)], [1352], level_res=[1352], tile=8)


def test_candidates_in_global_memory(env):
    # 234 k axis pixels, all of the same width
    _check(env, [_problem(_comb(600), 40, 600)], [600], level_res=[600], tile=8)


@pytest.mark.parametrize("rings,grid", [(_star(), 1352), (_comb(480), 480)])
def test_more_elements_than_ranked(env, rings, grid):
    # beyond 4096 elements the next one is found step by step; 21 k axis pixels in shared memory, 149 k in global
    prob = _problem(rings, 4100, grid)
    col = env[1](prob, level_res=[grid], tile=8)
    axis, width = (m.cpu().numpy() for m in col.mat_init(want_maps=True))
    assert np.array_equal(col.get_params().cpu().numpy(), _greedy(prob, axis, width, grid))
    col.close()


def test_both_forms_in_a_batch(env):
    probs = [_problem(_star(), 30, 1352), _problem(_star(), 30, 336), _problem(_star(), 9, 1352, seed=5)]
    _check(env, probs, [1352, 336, 1352], n_levels=1, level_res=[1], tile=8)
