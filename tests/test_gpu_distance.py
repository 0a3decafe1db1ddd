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
