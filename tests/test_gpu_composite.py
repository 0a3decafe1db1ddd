"""The composite's runs of tiles against the FP64 oracle: levels large and sparse enough that a warp takes
many tiles at once (most without coverage), both tile sides, and more problems than one round of loads
over the lanes places."""
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


@pytest.mark.parametrize("tile", [8, 16])
@pytest.mark.parametrize("gamma", [5e-4, 0.0])
def test_sparse_large_level(env, tile, gamma):
    O, Collage = env
    R = 1500  # ragged for both tiles
    prob = W.config_problem(2, n_elems=6, grid=R)
    g, o = U.paired(gamma=gamma, pad_px=1.0)
    col = Collage(prob, level_res=[R], tile=tile, **g)
    sc, q = O.Scene(prob), prob["params0"].astype(np.float64)
    ref = sc.eval(q, R, o)
    ihat, atau, _ = sc.render(q, R, o)
    for _ in range(2):  # the images of a render and of an iteration do not disturb one another
        bw, tau = (x.cpu().numpy().reshape(R, R) for x in col.render())
        assert np.abs(bw - ihat).max() <= U.COV_ATOL and np.abs(tau - atau).max() <= U.COV_ATOL
        terms, grad = col.loss_backward()
        U.check_terms(terms.cpu().numpy()[0], ref["terms"], R, (3e3, 8e4, gamma, 0.0), use_u=gamma != 0)
        U.check_grad(grad.cpu().numpy(), ref["grad_a"])
    col.close()


def test_more_than_1024_problems(env):
    O, Collage = env
    n = 1030
    probs = [W.config_problem(2, i, n_elems=1 + i % 3, grid=(16, 40)[i % 2]) for i in range(n)]
    g, o = U.paired()
    col = Collage(probs, level_res=[1], tile=8, **g)
    bw, _ = col.render()
    terms, _ = col.loss_backward()
    bw, terms = bw.cpu().numpy(), terms.cpu().numpy()
    off = 0
    for i, p in enumerate(probs):
        R = p["grid"]
        if i in (0, 1, 31, 32, 1023, 1024, n - 1):
            q = p["params0"].astype(np.float64)
            ihat, _, _ = O.Scene(p).render(q, R, o)
            assert np.abs(bw[off:off + R * R].reshape(R, R) - ihat).max() <= U.COV_ATOL
            U.check_terms(terms[i], O.Scene(p).eval(q, R, o)["terms"], R, (3e3, 8e4, 5e-4, 0.0))
        off += R * R
    col.close()
