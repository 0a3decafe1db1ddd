"""The loss of a problem assembled by several blocks against the FP64 oracle: one part, two, an uneven last
one, the most, and beside a problem too small to fill its parts; with the distribution term (whose adjoint
the sums do not wait for) and without."""
import numpy as np
import pytest

from paper_2406_04008_gb300 import workloads as W
from tests import _util as U

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("gamma", [5e-4, 0.0])
@pytest.mark.parametrize("sizes", [(360,), (520,), (730,), (1460,), (16, 900)])
def test_terms_by_parts(oracle_mod, sizes, gamma):
    from paper_2406_04008_gb300 import build
    build.build()
    from paper_2406_04008_gb300.collage import Collage
    O = oracle_mod
    probs = [W.config_problem(2, i, n_elems=8, grid=R) for i, R in enumerate(sizes)]
    g, o = U.paired(gamma=gamma)
    col = Collage(probs, level_res=[1], tile=8, **g)
    first = None
    for _ in range(4):  # plain launches, then one graph; the same sums each time
        terms = col.loss_backward()[0].cpu().numpy()
        first = terms if first is None else first
        assert (terms == first).all()
    for i, (p, R) in enumerate(zip(probs, sizes)):
        ref = O.Scene(p).eval(p["params0"].astype(np.float64), R, o)["terms"]
        U.check_terms(terms[i], ref, R, (3e3, 8e4, gamma, 0.0), use_u=gamma != 0)
    col.close()
