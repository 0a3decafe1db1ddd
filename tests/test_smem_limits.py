"""The shared-memory limit that a distance-transform kernel asks for is one figure, whatever the side: it is
an attribute of the function on the device, and with a figure per call a smaller call on another thread
would lower it between a larger one's setting and its launch.  (No GPU: the runtime's calls are recorded
by a stand-in, and the launches fail.)"""
import os
import subprocess

import pytest

from paper_2406_04008_gb300 import build

SRC = """
#include <cuda_runtime.h>
#include <cstdio>
#include <map>
#include <set>
static std::map<const void*, std::set<int>> g_limits;
template <class F>
static cudaError_t fake_set(F* f, cudaFuncAttribute, int v) {
  g_limits[(const void*)f].insert(v);
  return cudaSuccess;
}
#define cudaFuncSetAttribute fake_set
#define cudaMemsetAsync(...) cudaSuccess
#include "FILE"
int main() {
  using namespace collage;
  Dev d{};
  d.n_probs = d.total_tiles = 1;
  d.tile = 8;
  for (int side : {64, 12544, 16384, 17920, 32768}) CALL;
  size_t most = 0;
  for (auto& l : g_limits) {
    for (int v : l.second) printf("%d ", v);
    printf("\\n");
    most = l.second.size() > most ? l.second.size() : most;
  }
  return g_limits.empty() ? 2 : most > 1;
}
"""


@pytest.mark.parametrize("file,call", [
    ("mat.cu", "launch_mat_init(d, 0, side, 0, 0, 0, 0, 0, 0, 0, 0)"),
    ("metrics.cu", "launch_metrics(d, 0, 0, 0, 0, 0, side)"),
])
def test_one_limit_per_kernel(tmp_path, file, call):
    src, exe = tmp_path / "t.cu", str(tmp_path / "t")
    src.write_text(SRC.replace("FILE", file).replace("CALL", call))
    subprocess.run([build._nvcc(), *build.ARCH, "-std=c++17", "-O0", "-I" + build.INCLUDE, "-I" + build.CSRC, str(src),
                    "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True, env=dict(os.environ, CUDA_VISIBLE_DEVICES=""))
    assert r.returncode == 0, r.stdout
