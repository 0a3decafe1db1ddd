"""Buffers that a kernel must not take: too few floats, and memory that is not the handle's device's (no
GPU: nothing is launched); and the calls that choose between a kernel and a copy, in a captured graph."""
import os
import subprocess

import numpy as np
import pytest
import torch

from paper_2406_04008_gb300 import build, collage
from paper_2406_04008_gb300 import workloads as W
from tests import _util as U

CUDA = os.environ.get("CUDA_HOME", "/usr/local/cuda")


class _OnDevice:
    """What the binding asks of a CUDA tensor."""

    dtype, is_cuda = torch.float32, True

    def __init__(self, n):
        self.n = n

    def detach(self):
        return self

    def is_contiguous(self):
        return True

    def numel(self):
        return self.n

    def data_ptr(self):
        return 1 << 20


class _Lib:
    calls = 0

    def collage_set_params(self, h, stream, ptr):
        self.calls += 1
        return 0


@pytest.mark.parametrize("n,taken", [(0, 0), (4, 0), (11, 0), (12, 1), (16, 1)])
def test_set_params_counts_its_floats(monkeypatch, n, taken):
    monkeypatch.setattr(collage, "_stream", lambda: 0)
    col = collage.Collage.__new__(collage.Collage)
    col.lib, col.h, col.n_elems = _Lib(), None, 3
    if taken:
        col.set_params(_OnDevice(n))
    else:
        with pytest.raises(ValueError):
            col.set_params(_OnDevice(n))
    assert col.lib.calls == taken


def test_kernels_take_the_handles_own_memory_only(tmp_path):
    src = tmp_path / "route.cpp"
    src.write_text("""#include "route.h"
int main() {
  using collage::kernel_route;
  const cudaMemoryType other[] = {cudaMemoryTypeUnregistered, cudaMemoryTypeHost, cudaMemoryTypeManaged};
  int bad = !kernel_route(cudaMemoryTypeDevice, 0, 0) || !kernel_route(cudaMemoryTypeDevice, 3, 3);
  bad |= kernel_route(cudaMemoryTypeDevice, 1, 0) || kernel_route(cudaMemoryTypeDevice, 0, 1);
  for (cudaMemoryType t : other) bad |= kernel_route(t, 0, 0);
  return bad;
}
""")
    exe = str(tmp_path / "route")
    subprocess.run(["g++", "-std=c++17", "-I" + os.path.join(CUDA, "include"), "-I" + build.CSRC, str(src), "-o", exe],
                   check=True)
    assert subprocess.run([exe]).returncode == 0


@pytest.mark.gpu
def test_params_in_and_out_of_a_captured_graph():
    # whose memory a pointer is gets asked while the caller's stream is captured
    build.build()
    prob = W.config_problem(2, n_elems=20, grid=128)
    g, _ = U.paired()
    g.update(level_res=[128], tile=8, deterministic=1, use_graphs=0)  # (a graph launch can not be captured)
    a, b = collage.Collage(prob, **g), collage.Collage(prob, **g)
    q = torch.from_numpy(prob["params0"].reshape(-1, 4).copy()).cuda()
    for h in (a, b):
        h.step(1)  # sizes settled
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        a.set_params(q)
        a.step_async(2)
        out = a.get_params()
    for k in range(3):
        q[:, 2] += 0.1
        graph.replay()
        b.set_params(q)
        b.step(2)
        assert torch.equal(out, b.get_params()) and np.isfinite(out.cpu().numpy()).all(), k
    a.close()
    b.close()
