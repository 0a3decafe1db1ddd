"""Overlapped launches against plain stream order: the adjoint reads what earlier kernels of the iteration
wrote while its predecessor drains, so every iteration of a run has to see its own images, lists and
segments.  Bit for bit over runs of many iterations, in which all of them change."""
import numpy as np
import pytest

from paper_2406_04008_gb300 import workloads as W
from tests import _util as U

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("config,n,R,tile,graphs", [
    (2, 40, 256, 8, 1), (2, 40, 256, 16, 0), (3, 300, 512, 8, 0), (3, 1000, 1024, 8, 1), (2, 12, 1000, 16, 1)])
def test_overlapped_iterations_equal_plain_ones(config, n, R, tile, graphs):
    from paper_2406_04008_gb300 import build
    build.build()
    from paper_2406_04008_gb300.collage import Collage
    prob = W.config_problem(config, n_elems=n, grid=R)
    g, _ = U.paired(pad_px=1.0)
    out = []
    for overlap in (1, 0):
        col = Collage(prob, level_res=[R], tile=tile, deterministic=1, use_graphs=graphs, overlap_launches=overlap, **g)
        q = []
        for _ in range(6):
            col.step(40)
            q.append(col.get_params().cpu().numpy())
        out.append((np.stack(q), col.loss().cpu().numpy()))
        col.close()
    (qa, la), (qb, lb) = out
    assert np.array_equal(qa, qb) and np.array_equal(la, lb)
    assert np.abs(qa[-1] - qa[0]).max() > 0.01
