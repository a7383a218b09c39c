"""The Phase-3 kernel that a solve runs by default, checked on the host (no GPU).

`solve_phase3` in `csrc/fw_launch.h` turns the default table's single launch into one launch per round where that is
faster.  This test copies both functions out of the header unchanged, compiles them with g++ and compares them with
the ranges that `include/apsp.h` documents at `apsp_tuned_config`.
"""
import os
import re
import shutil
import subprocess

import pytest

from tests.test_plan_source import CSRC, ROOT, _block

MAIN = r"""
#include <cstdio>
#include <cstdlib>
int main(int argc, char **argv) {
  for (int i = 1; i < argc; ++i)
    for (int dt = 0; dt < 3; ++dt)
      printf("%s %d %d %d\n", argv[i], dt, apsp::default_phase3(atoll(argv[i]), dt),
             apsp::solve_phase3(atoll(argv[i]), dt));
}
"""


def test_solves_follow_the_documented_ranges(tmp_path):
    if shutil.which("g++") is None:
        pytest.skip("g++ needed")
    hdr = open(os.path.join(CSRC, "fw_launch.h")).read()
    doc = re.sub(r"\s*\*\s*", " ", open(os.path.join(ROOT, "include", "apsp.h")).read())
    m = re.search(r"int32 below n = (\d+) and from (\d+), packed 16-bit below (\d+) and from (\d+), fp32 at every n",
                  doc)
    lo0, hi0, lo1, hi1 = (int(x) for x in m.groups())
    prog = "\n".join(["#include <cstdint>", "namespace apsp {",
                      _block(hdr, "inline int default_phase3(", with_template=False),
                      _block(hdr, "inline int solve_phase3(", with_template=False), "}", MAIN])
    src, exe = tmp_path / "route.cpp", tmp_path / "route"
    src.write_text(prog)
    subprocess.run(["g++", "-O2", "-std=c++17", "-o", str(exe), str(src)], check=True)
    ns = sorted({1, 64, 4096, 6143, 6144, 24575, 24576, 49151, 49152, 65536, 262144}
                | {x + d for x in (lo0, hi0, lo1, hi1) for d in (-1, 0, 1)})
    out = subprocess.run([str(exe)] + [str(n) for n in ns], check=True, capture_output=True, text=True).stdout
    for line in out.splitlines():
        n, dt, table, run = (int(x) for x in line.split())
        single = (lo0 <= n < hi0, lo1 <= n < hi1, False)[dt]
        assert run == (4 if single and table == 4 else 3), (n, dt)
        assert not single or table == 4, (n, dt)  # the ranges lie inside the table's
