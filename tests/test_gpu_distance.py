"""The exact distance transform behind the quality metrics and the skeleton-based initialisation, and
the placement, at the sizes where their passes have edges: sides about the 8-row bytes and 32-row
words of the column pass, and more axis pixels than the placement keeps in shared memory."""
import numpy as np
import pytest
import torch

from paper_2406_04008_gb300 import workloads as W
from tests import _util as U
from tests.test_gpu_mat import _check as check_mat
from tests.test_gpu_parity import _check_metrics

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env(oracle_mod):
    from paper_2406_04008_gb300 import build
    build.build()
    from paper_2406_04008_gb300.collage import Collage
    assert torch.cuda.is_available()
    return oracle_mod, Collage


@pytest.mark.parametrize("grid", [31, 32, 33, 65, 257])
def test_metrics_at_word_edges(env, grid):
    # no pixel of these cases lies within 1e-4 of a threshold: the counts are exact, and L-nU (sums of
    # integers) agrees to rounding
    O, Collage = env
    prob = W.config_problem(2, n_elems=12, grid=grid)
    g, o = U.paired()
    col = Collage(prob, level_res=[grid], tile=8, **g)
    _check_metrics(col.metrics()[0], O.Scene(prob).metrics(prob["params0"].astype(np.float64), grid, o), 0)
    col.close()


def test_metrics_without_objects(env):
    # every element off the image: no object pixel in any column
    O, Collage = env
    prob = W.config_problem(2, n_elems=3, grid=65)
    prob["params0"][0::4] += 4.0
    g, o = U.paired()
    col = Collage(prob, level_res=[65], tile=8, **g)
    m = col.metrics()[0]
    assert m[0] == m[2] == m[3] == m[7] == 0.0 and m[1] > 0
    col.close()


@pytest.mark.parametrize("grid", [31, 32, 33, 65, 257])
def test_mat_init_at_word_edges(env, grid):
    check_mat(env, [W.config_problem(2, n_elems=12, grid=grid)], [grid], level_res=[grid], tile=8)


def test_mat_init_candidates_in_global_memory(env):
    # 16484 axis pixels: more than 512 groups of 32
    check_mat(env, [W.config_problem(3, n_elems=30, grid=1100)], [1100], level_res=[1100], tile=8)


@pytest.mark.parametrize("tile", [8, 16])
def test_container_rings_far_and_crossing(env, tile):
    # the container raster picks each tile's segments: a ring whose edges pass far outside the image on
    # every side (only the winding of the tiles shows it), a hole across many tiles, and rings left
    # and right of the image (neither, or only, crossed by the tiles' rays)
    rng = W.PCG32(12)
    hole = W.star_container(rng, r_in=0.11, r_out=0.31)[0][::-1]
    far = np.array([(-40.0, -30.0), (60.0, -31.0), (61.0, 45.0), (-41.0, 44.0)])
    left = W.regular_polygon(0.4, 7) + (-1.5, 0.5)
    right = W.regular_polygon(0.4, 9) + (2.5, 0.45)
    els = [(1, W.regular_polygon(0.02 + 0.01 * k, 6), 0.0) for k in range(4)]
    params = [(0.2 + 0.1 * k, 0.3, 0.1 * k, 1.0) for k in range(4)]
    prob = W.make_problem(els, [far, hole, left, right], params, 200)
    check_mat(env, [prob], [200], level_res=[200], tile=tile)
