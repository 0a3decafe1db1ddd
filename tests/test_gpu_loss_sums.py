"""The overlap loss against its own pixels: the mean of max(0, A - tau) over the rendered A in FP64.  A loss term
is a sum of non-negative floats kept in 1024 accumulators and then in float pairs, and rounded once: half an
ulp (2^-24 of the value), and a quarter of that for the accumulators' own roundings, which are independent and
of which each touches a thousandth of the sum."""
import numpy as np
import pytest

from paper_2406_04008_gb300 import workloads as W
from tests import _util as U

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("R", [120, 333, 512, 1000, 1024])  # one part, several, the most
@pytest.mark.parametrize("tile", [8, 16])
def test_overlap_loss_is_rounded_once(R, tile):
    from paper_2406_04008_gb300 import build
    build.build()
    from paper_2406_04008_gb300.collage import Collage
    g, o = U.paired(pad_px=2.0)
    off = []
    for index in range(4):
        prob = W.config_problem(2, collage_index=index, n_elems=60, grid=R)
        col = Collage(prob, level_res=[R], tile=tile, **g)
        _, tau = col.render()
        terms, _ = col.loss_backward()
        a = tau.cpu().numpy() - np.float32(o.tau)  # (exact: A lies within a factor 2 of tau, or below it)
        exact = np.maximum(a, 0).astype(np.float64).mean()
        off.append(abs(float(terms[0, 1]) / exact - 1.0))
        t = terms[0].cpu().numpy().astype(np.float64)
        total = 3e3 * t[0] + 8e4 * t[1] + float(np.float32(5e-4)) * t[2]
        assert abs(t[4] / total - 1.0) <= 2.0 * 2.0 ** -24  # (its terms and itself, rounded once each)
        col.close()
    assert max(off) <= 1.25 * 2.0 ** -24, off
