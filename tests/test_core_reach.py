"""The reach of the restriction stencils behind the core lists (CORE_HOPS in
csrc/sww_core.cuh): everything the restriction to a coarser level reads is owned by a
node within two hops of a point that is live there, for every coarse edge of the
library's own host tables (tests/core_reach_check.cpp; no GPU).  A divergence reads the
fluxes of its node's ring, one hop further: three."""
import os
import re
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1404_0405_gb300", "csrc")


def test_restriction_reach(tmp_path):
    exe = str(tmp_path / "core_reach_check")
    subprocess.run(["g++", "-O2", "-std=c++17", "-fopenmp", "-I", CSRC, os.path.join(CSRC, "grid.cpp"),
                    os.path.join(ROOT, "tests", "core_reach_check.cpp"), "-o", exe], check=True)
    reach = int(subprocess.run([exe, "2", "6"], check=True, capture_output=True, text=True).stdout)
    hops = int(re.search(r"CORE_HOPS = (\d+);", open(os.path.join(CSRC, "sww_core.cuh")).read()).group(1))
    assert reach == 2 and hops >= reach + 1
