"""A replayed loss + gradient pass whose pairs outgrow the captured buffers: the buffers grow, the pass runs
again and agrees with eager launches bit for bit, and later passes are captured anew."""
import pytest
import torch

from tests.test_gpu_grad_graph import Collage, _pair  # noqa: F401  (the fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("level", [0, 1])
def test_replay_outgrows_its_buffers(Collage, level):  # noqa: F811
    prob, a, b = _pair(Collage)
    q0 = torch.from_numpy(prob["params0"].reshape(-1, 4).copy()).cuda()
    big = q0.clone()
    big[:, 3] = 6.0
    for h in (a, b):
        h.set_level(level)
    cap = a.info()["pair_capacity"]
    for i in range(12):
        q = big if i >= 6 else q0
        for h in (a, b):
            h.set_params(q)
        (ta, ga), (tb, gb) = a.loss_backward(), b.loss_backward()
        assert torch.equal(ta, tb) and torch.equal(ga, gb), i
        if i < 6:
            assert a.info()["pair_capacity"] == cap
        else:
            assert a.info()["pair_capacity"] > cap and a.info()["last_pairs"] > cap
    a.close()
    b.close()
