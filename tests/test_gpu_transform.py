"""The transform's float-pair rotation against the FP64 oracle: angles on both sides of the range the
pairs cover, and element counts on both sides of the four-elements-per-block form."""
import numpy as np
import pytest
import torch

from paper_2406_04008_gb300 import workloads as W
from tests import _util as U

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env(oracle_mod):
    from paper_2406_04008_gb300 import build
    build.build()
    from paper_2406_04008_gb300.collage import Collage
    assert torch.cuda.is_available()
    return oracle_mod, Collage


def _check(env, prob, grid):
    O, Collage = env
    g, o = U.paired(gamma=0.0)
    col = Collage(prob, level_res=[grid], tile=8, **g)
    bw, tau = (x.cpu().numpy().reshape(grid, grid) for x in col.render())
    terms, grad = col.loss_backward()
    sc, q = O.Scene(prob), prob["params0"].astype(np.float64)
    ihat, atau, _ = sc.render(q, grid, o)
    assert np.abs(bw - ihat).max() <= U.COV_ATOL and np.abs(tau - atau).max() <= U.COV_ATOL
    ref = sc.eval(q, grid, o)
    U.check_terms(terms.cpu().numpy()[0], ref["terms"], grid, (3e3, 8e4, 0.0, 0.0), use_u=False)
    U.check_grad(grad.cpu().numpy(), ref["grad_a"])
    col.close()


def test_angles(env):
    prob = W.config_problem(2, n_elems=12, grid=128)
    prob["params0"][2::4] = [0.0, -0.0, 1e-30, np.pi, -np.pi / 2, 100.0, 8191.5, 8192.0, -8192.0, 8193.0, -3e4, 1e6]
    _check(env, prob, 128)


@pytest.mark.parametrize("n", [4095, 4096, 4097])
def test_element_counts(env, n):
    rng = W.PCG32(31)
    els, params = [], []
    for _ in range(n):
        els.append((1, W.regular_polygon(0.004 + 0.004 * rng.uniform(), 5), 0.0))
        params.append((rng.uniform(), rng.uniform(), 6.0 * rng.uniform(), 0.8 + 0.4 * rng.uniform()))
    _check(env, W.make_problem(els, W.disk_container(), params, 512), 512)
