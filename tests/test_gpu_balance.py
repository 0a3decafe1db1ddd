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


@pytest.mark.parametrize("n_dil,emit,R,copies", [(1, 256, 1000, 5), (8, 256, 1000, 5), (8, 128, 600, 9), (1, 256, 250, 30)])
def test_every_kernel_count_and_block_size(n_dil, emit, R, copies):
    # the distribution term's grids beyond what is resident at once (two blocks an SM for the adjoint of eight
    # kernels), its listed tiles on both sides of the limit, and the emission's wide blocks
    from paper_2406_04008_gb300 import build
    build.build()
    from paper_2406_04008_gb300.collage import Collage
    prob = W.config_problem(2, n_elems=60, grid=R)
    g, _ = U.paired(n_dil=n_dil, dil_weight=tuple(1.0 + k for k in range(8)))

    def steps(problems, **kw):
        col = Collage(problems, level_res=[R], tile=8, deterministic=True, **g, **kw)
        col.set_tuning(emit_threads=emit, chunk_px=64)
        col.step(3)
        q, (terms, _) = col.get_params().cpu().numpy().reshape(len(problems), -1), col.loss_backward()
        terms = terms.cpu().numpy()
        col.close()
        return q, terms

    alone, t1 = steps([prob])
    many, tm = steps([prob] * copies)
    assert (many == alone).all() and (tm == t1).all() and t1[0, 2] > 0
    plain, tp = steps([prob], persistent=False, overlap_launches=0)
    assert (plain == alone).all() and (tp == t1).all()
