"""The stages whose release a converter group waits for before its CTA leaves (stage_drain.h),
compiled for the host: together the groups must see every slot's last stage, and each of them."""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2606_11536_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <set>
#include "stage_drain.h"
int main() {
  for (uint32_t ring = 1; ring <= 6; ++ring)
    for (uint32_t groups = 1; groups <= ring; ++groups)
      for (uint64_t stages = 0; stages <= 50; ++stages) {
        std::set<uint64_t> want, got;
        for (uint64_t g = stages > ring ? stages - ring : 0; g < stages; ++g) want.insert(g);
        for (uint32_t group = 0; group < groups; ++group)
          for (uint64_t g = gbpir::first_undrained(stages, group, groups, ring); g < stages; g += groups)
            if (g % groups != group || !got.insert(g).second) return 2;
        if (got != want) {
          std::printf("ring %u, %u groups, %llu stages\n", ring, groups, (unsigned long long)stages);
          return 1;
        }
      }
  return 0;
}
"""


def test_every_slots_last_release_is_waited_for(tmp_path):
    src = tmp_path / "drain.cc"
    src.write_text(PROGRAM)
    exe = tmp_path / "drain"
    subprocess.run(["g++", "-std=c++17", "-Wall", "-Werror", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout


def test_the_converters_use_the_rule():
    for name in ("gemm_digit.cu", "lwe_tc.cu"):
        assert "g = first_undrained(stages, group, " in open(os.path.join(CSRC, name)).read(), name
