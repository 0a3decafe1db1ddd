"""Blocks that take their work by rank on their SM against blocks that take it by index: a problem whose
grids fit the device at once, iterated alone, ends with the very params that it has among copies too many
for that (deterministic gradients, one launch configuration)."""
import numpy as np
import pytest

from paper_2406_04008_gb300 import workloads as W
from tests import _util as U

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("R,n,copies,tile,config", [
    (16, 1, 1400, 8, 2),    # one block of each grid has work
    (72, 24, 140, 8, 2),    # 9 tiles of the distribution term of 152 and more
    (200, 120, 30, 16, 3),
    (1000, 300, 5, 8, 2),   # the largest balanced grid of the distribution term, its last range partial
])
def test_alone_and_among_copies(R, n, copies, tile, config):
    from paper_2406_04008_gb300 import build
    build.build()
    from paper_2406_04008_gb300.collage import Collage
    prob = W.config_problem(config, n_elems=n, grid=R)
    g, _ = U.paired()

    def steps(problems, **kw):
        col = Collage(problems, level_res=[R], tile=tile, deterministic=True, **g, **kw)
        col.set_tuning(emit_threads=128, chunk_px=64)
        for k in (1, 1, 3):
            col.step(k)
        q, (terms, _) = col.get_params().cpu().numpy().reshape(len(problems), -1), col.loss_backward()
        terms = terms.cpu().numpy()
        col.close()
        return q, terms

    alone, t1 = steps([prob])
    assert np.isfinite(alone).all() and np.abs(alone[0] - prob["params0"].reshape(-1)).max() > 0
    many, tm = steps([prob] * copies)
    assert (many == alone).all() and (tm == t1).all()
    by_index, ti = steps([prob], persistent=False)
    assert (by_index == alone).all() and (ti == t1).all()
