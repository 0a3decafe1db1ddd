"""The emission's shape across levels: it follows each level's work in an untuned handle and beside a search's
choice, which holds at the level it was timed at; a shape that the caller sets holds at every level."""
import pytest

from paper_2406_04008_gb300 import workloads as W
from tests import _util as U

pytestmark = pytest.mark.gpu

SHAPE = ("emit_threads", "chunk_px")


def _handle(tile=8):
    from paper_2406_04008_gb300 import build
    build.build()
    from paper_2406_04008_gb300.collage import Collage
    # 40 elements that are one chunk each at 128^2 and ten at 1024^2
    prob = W.config_problem(2, n_elems=40, grid=1024)
    prob["params0"][3::4] *= 3.0
    g, _ = U.paired()
    return Collage(prob, tile=tile, n_levels=2, level_res=[128, 1024], level_iters=[1, 1], **g)


def _shapes(col):
    out = []
    for level in (0, 1, 0, 1):
        col.set_level(level)
        t = col.tuning()
        out.append(tuple(t[k] for k in SHAPE))
    assert out[:2] == out[2:]
    return out[:2]


def test_a_search_leaves_the_other_levels_to_their_work():
    untuned = {}
    for tile in (8, 16):
        plain = _handle(tile)
        untuned[tile] = _shapes(plain)
        assert untuned[tile][0] != untuned[tile][1]
        plain.close()
    for from_cache in (0, 1):
        col = _handle()
        col.set_level(1)
        col.autotune()
        t = col.tuning()
        assert t["from_cache"] == from_cache
        at1 = tuple(t[k] for k in SHAPE)
        assert _shapes(col) == [untuned[t["tile"]][0], at1]
        col.run_schedule()
        assert tuple(col.tuning()[k] for k in SHAPE) == at1
        col.close()


def test_a_set_shape_holds_at_every_level():
    col = _handle()
    for shape in ((128, 64), (256, 32)):
        col.set_tuning(emit_threads=shape[0], chunk_px=shape[1])
        assert _shapes(col) == [shape, shape]
    col.close()
