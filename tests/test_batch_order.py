"""CPU check of the weight that orders a batch's chunk queue: the sweeps a chunk
runs, which since the frozen ones are cut short differ between noise classes with
the same schedule length."""
import subprocess

from paper_2509_17837_gb300 import build

PROGRAM = r"""
#include "batch_internal.h"
#include <cstdio>
int main() {
  const int rows[][3] = {{21, 2000, 400}, {21, 2000, 1500}, {21, 2000, 2000}, {21, 500, 500}, {17, 2000, 1500}, {21, 0, 0}};
  for (const auto& r : rows) {
    xzzx::batch::ChunkDev c{};
    c.d = r[0], c.n_sweeps = r[1], c.n_live = r[2];
    std::printf("%lld\n", (long long)xzzx::batch::chunk_work(c));
  }
}
"""


def test_chunks_weigh_the_sweeps_they_run(tmp_path):
    (tmp_path / "order.cu").write_text(PROGRAM)
    exe = str(tmp_path / "order")
    subprocess.run([build.nvcc(), str(tmp_path / "order.cu"), "-o", exe] + build.NVCC_FLAGS, check=True)
    short, longer, whole, few, smaller, none = map(int, subprocess.run([exe], capture_output=True, text=True,
                                                                       check=True).stdout.split())
    assert short < longer < whole == 2000 * (21 * 21 - 1)
    assert 400 * 440 < short < 600 * 440  # its live sweeps and the few until its chains repeat
    assert few == 500 * 440 and smaller < longer and none == 0
