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
