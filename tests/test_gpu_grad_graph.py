"""The graph behind repeated loss + gradient passes: the same numbers as eager launches, bit for bit in
deterministic mode, across new params, a level change and a bin overflow between passes; and the one-launch
forms of set_params / get_params beside the copies that unaligned buffers take."""
import numpy as np
import pytest
import torch

from paper_2406_04008_gb300 import workloads as W
from tests import _util as U

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def Collage():
    from paper_2406_04008_gb300 import build
    build.build()
    from paper_2406_04008_gb300.collage import Collage as C
    return C


def _pair(Collage, **kw):
    prob = W.config_problem(2, n_elems=30, grid=256)
    g, _ = U.paired(pad_px=1.0)
    g.update(level_res=[128, 256], level_iters=[1, 1], n_levels=2, tile=8, deterministic=1, **kw)
    return prob, Collage(prob, use_graphs=1, **g), Collage(prob, use_graphs=0, **g)


def test_graph_passes_equal_eager_passes(Collage):
    prob, a, b = _pair(Collage)
    q0 = torch.from_numpy(prob["params0"].reshape(-1, 4).copy()).cuda()
    for level in (0, 1, 0):
        a.set_level(level)
        b.set_level(level)
        for i in range(6):  # eager passes, the capture, replays
            q = q0.clone()
            q[:, :2] += 0.01 * torch.sin(torch.arange(len(q), device="cuda") + i)[:, None]
            if i == 4:  # enlarged behind the captured capacity: the pass overflows, regrows and runs again
                q[:, 3] = 2.5
            a.set_params(q)
            b.set_params(q)
            ta, ga = a.loss_backward()
            tb, gb = b.loss_backward()
            assert torch.equal(ta, tb) and torch.equal(ga, gb), (level, i)
            assert torch.equal(a.get_params(), q)
    a.close()
    b.close()


def test_graph_pass_after_a_step(Collage):
    # a pending Adam step is applied by the pass that follows, in a replay as in an eager one
    _, a, b = _pair(Collage)
    for _ in range(4):
        for h in (a, b):
            h.step(1)
        ta, ga = a.loss_backward()
        tb, gb = b.loss_backward()
        assert torch.equal(ta, tb) and torch.equal(ga, gb)
    assert torch.equal(a.get_params(), b.get_params())
    a.close()
    b.close()


def test_unaligned_param_buffers(Collage):
    prob, a, b = _pair(Collage)
    n = a.n_elems * 4
    q = torch.from_numpy(prob["params0"].copy()).cuda() + 0.001
    buf = torch.empty(n + 1, device="cuda")
    buf[1:] = q
    for h, src in ((a, buf[1:]), (b, q)):  # 4 bytes past a 16-byte boundary; on one
        h.step(1)  # a step is pending
        h.set_params(src)
    assert torch.equal(a.get_params().reshape(-1), q) and torch.equal(b.get_params().reshape(-1), q)
    a.step(1)
    b.step(1)
    out = torch.zeros(n + 1, device="cuda")
    assert a.lib.collage_get_params(a.h, torch.cuda.current_stream().cuda_stream, out[1:].data_ptr()) == 0
    assert torch.equal(out[1:], b.get_params().reshape(-1)) and out[0] == 0
    a.close()
    b.close()
