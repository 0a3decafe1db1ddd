"""Sides whose rows need more than 48 KB of shared memory in the distance transform: the limits that two
handles' calls need do not disturb one another."""
import threading

import numpy as np
import pytest
import torch

from paper_2406_04008_gb300 import workloads as W
from tests import _util as U

pytestmark = pytest.mark.gpu


def test_two_large_sides_on_two_threads():
    from paper_2406_04008_gb300 import build
    build.build()
    from paper_2406_04008_gb300.collage import Collage
    g, _ = U.paired(gamma=0.0)
    sides, cols = (12544, 17920), []
    for R in sides:
        rng = W.PCG32(2)
        els = [(1, W.regular_polygon(0.002 + 0.001 * k, 7), 0.0) for k in range(3)]
        params = [(0.3 + 0.2 * rng.uniform(), 0.4, 0.1, 1.0) for _ in els]
        # a small container: the passes' own work is not the point
        prob = W.make_problem(els, [W.regular_polygon(0.01, 64) + (0.5, 0.5)], params, R)
        cols.append(Collage(prob, level_res=[R], tile=16, **g))
    faults, results, start = [], {}, threading.Barrier(2)

    def run(R, col):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                start.wait()
                for _ in range(40):
                    for _ in range(10):
                        col.mat_init()
                    torch.cuda.current_stream().synchronize()
                results[R] = col.get_params().cpu().numpy()
        except Exception as e:
            faults.append((R, str(e)))

    threads = [threading.Thread(target=run, args=a) for a in zip(sides, cols)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not faults, faults
    for R in sides:  # the widest pixel: one of those about the container's centre
        assert np.abs(results[R][np.argmax([0.002, 0.003, 0.004]), :2] - 0.5).max() <= 2.0 / R
    m = cols[1].metrics()
    assert np.isfinite(m).all() and m[0, 1] == pytest.approx(np.pi * 0.01 ** 2 * sides[1] ** 2, rel=0.01)
    for c in cols:
        c.close()
