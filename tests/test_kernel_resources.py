"""CPU check of what the compiler makes of the persistent annealing kernels: the
several distances of one kernel share its register bound and none of them spills
(a spill inside a sweep costs 10 to 40% of a batch that does not fill the GPU)."""
import concurrent.futures as cf
import os
import re
import subprocess

from paper_2509_17837_gb300 import build


def ptxas_report(unit, tmp):
    cmd = [build.nvcc(), "-c", os.path.join(build.CSRC, unit + ".cu"), "-o", str(tmp / (unit + ".o")), "-Xptxas", "-v"]
    r = subprocess.run(cmd + build.NVCC_FLAGS, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return r.stdout + r.stderr


def test_persistent_kernels_do_not_spill(tmp_path):
    units = ["batch_persist%d_nt128_u1" % dmax for dmax in (15, 21, 31)]
    with cf.ThreadPoolExecutor(len(units)) as ex:
        reports = list(ex.map(lambda u: ptxas_report(u, tmp_path), units))
    for unit, text in zip(units, reports):
        spills = re.findall(r"(\d+) bytes spill stores, (\d+) bytes spill loads", text)
        assert spills and all(s == ("0", "0") for s in spills), (unit, spills)


LANE_FORMS = r"""
#include "anneal_coop.cuh"
#include <cstdio>
using namespace xzzx::coop;
template <class G>
void forms(const char* name, int d) {
  const int per[4] = {Form<G, 1, 3, 3>::kPerSm, Form<G, 1, 3, 4>::kPerSm, Form<G, 4, 0, 3>::kPerSm, Form<G, 4, 0, 4>::kPerSm};
  const size_t bytes[4] = {Form<G, 1, 3, 3>::smem_bytes(64), Form<G, 1, 3, 4>::smem_bytes(64),
                           Form<G, 4, 0, 3>::smem_bytes(64), Form<G, 4, 0, 4>::smem_bytes(64)};
  for (int k = 0; k < 4; ++k) std::printf("%s %d %d %zu\n", name, d, per[k], bytes[k]);
}
template <int D>
void upto() {
  forms<RotLanes<D>>("rotated", D);
  forms<PlanarLanes<D>>("planar", D);
  if constexpr (D < 31) upto<D + 2>();
}
int main() { upto<3>(); }
"""


def test_lane_forms_fit_the_ctas_their_rules_count_on(tmp_path):
    """The launch rule sizes the lane-parallel forms for so many CTAs per SM: that
    many fit into an SM's 228 KB, with the kilobyte the system takes of each."""
    (tmp_path / "forms.cu").write_text(LANE_FORMS)
    exe = str(tmp_path / "forms")
    subprocess.run([build.nvcc(), str(tmp_path / "forms.cu"), "-o", exe] + build.NVCC_FLAGS, check=True)
    rows = [line.split() for line in subprocess.run([exe], capture_output=True, text=True, check=True).stdout.splitlines()]
    assert len(rows) == 2 * 15 * 4
    for lattice, d, per_sm, smem in rows:
        taken = -(-int(smem) // 128) * 128 + 1024
        assert int(per_sm) >= 3 and int(per_sm) * taken <= 228 * 1024, (lattice, d, per_sm, smem)
