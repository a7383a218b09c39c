"""What the request loop counts towards its memory budget, against what a batched plan takes (no GPU).

`BatchPlan::build` in `csrc/batch.cu` lays out the workspace of a group of requests, and `panel_bytes` in
`csrc/apsp_api.cu` is what each of them counts for.  This test copies both out of the sources unchanged, compiles
them with g++ and compares them: beyond the plan's small tables, a group takes no more than its requests count.
"""
import os
import re
import shutil
import subprocess

import pytest

from tests.test_plan_source import CSRC, _block

CUDA_INCLUDE = "/usr/local/cuda/include"

MAIN = r"""
#include <cstdio>
#include <cstdlib>
int main() {
  const int64_t ns[] = {1, 63, 64, 65, 100, 127, 128, 129, 255, 256, 257, 300, 511, 512, 513, 1000, 1535};
  for (int copy = 0; copy < 2; ++copy)
    for (size_t i = 0; i < sizeof(ns) / sizeof(ns[0]); ++i)
      for (int count : {1, 3, 64}) {
        std::vector<apsp::BatchInput> in;
        int64_t counted = 0;
        for (int g = 0; g < count; ++g) {
          const int64_t n = ns[(i + g) % (sizeof(ns) / sizeof(ns[0]))];
          const bool c = copy && n % 4 != 0;
          in.push_back(apsp::BatchInput{nullptr, nullptr, n, n, n, nullptr, c});
          counted += panel_bytes(n) + (c ? apsp::batch_copy_bytes(n) : 0);
        }
        apsp::BatchPlan plan;
        const size_t all = plan.build(in, nullptr);
        const size_t tables = apsp::pad256(plan.graphs.size() * sizeof(apsp::BatchGraph)) +
                              apsp::pad256(plan.segs.size() * sizeof(apsp::BatchSeg)) +
                              apsp::pad256(plan.ncounters * sizeof(int) + sizeof(unsigned long long));
        if ((int64_t)(all - tables) > counted) {
          printf("n %lld x %d copy %d: takes %zu, counts %lld\n", (long long)ns[i], count, copy, all - tables,
                 (long long)counted);
          return 1;
        }
      }
  return 0;
}
"""


def test_a_group_takes_no_more_than_its_requests_count(tmp_path):
    if shutil.which("g++") is None or not os.path.isdir(CUDA_INCLUDE):
        pytest.skip("g++ and the CUDA headers needed")
    batch = open(os.path.join(CSRC, "batch.cu")).read()
    panels = open(os.path.join(CSRC, "fw_panels.cuh")).read()
    api = open(os.path.join(CSRC, "apsp_api.cu")).read()
    prog = "\n".join([
        "#include <algorithm>", "#include <cstdint>", "#include <vector>", '#include "batch.h"', "namespace apsp {",
        "struct OpI32 { static constexpr int EPW = 1; };",
        re.search(r"constexpr int BK = \d+;", batch).group(0), re.search(r"constexpr int P2_XW = \d+;", batch).group(0),
        _block(panels, "struct alignas(16) DiagBuf {", with_template=False),
        _block(panels, "constexpr int64_t panel_chunks(").replace("__host__ __device__", ""),
        "inline " + _block(batch, "size_t pad256(size_t b)", with_template=False),
        _block(batch, "size_t BatchPlan::build(", with_template=False), "}",
        _block(api, "int64_t panel_bytes(int64_t n)", with_template=False), MAIN])
    src, exe = tmp_path / "budget.cpp", tmp_path / "budget"
    src.write_text(prog)
    subprocess.run(["g++", "-O1", "-std=c++17", f"-I{CSRC}", f"-I{CUDA_INCLUDE}", "-o", str(exe), str(src)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
