"""The autotuner's search, compiled from the sources with a timer of known
costs (no GPU): whatever schedule it starts from, it ends at the cheapest."""

import itertools
import os
import re
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

MAIN = r"""
#include <cstdio>
#include <cstdlib>
#include "ori.h"
%s
int main(int argc, char** argv) {
  // argv: mixed nv, start (7 fields), then 3 costs for each of the 7 fields
  const bool mixed = std::atoi(argv[1]) != 0;
  ori_schedule s{};
  int* f[7] = {&s.yfwd, &s.zconv, &s.yinv, &s.yfwd_variant, &s.zconv_variant, &s.yinv_variant, &s.ctas_per_sm};
  for (int i = 0; i < 7; ++i) *f[i] = std::atoi(argv[3 + i]);
  int calls = 0;
  auto time = [&](const ori_schedule& c, float* t) {
    const int v[7] = {c.yfwd, c.zconv, c.yinv, c.yfwd_variant, c.zconv_variant, c.yinv_variant, c.ctas_per_sm};
    *t = 0;
    for (int i = 0; i < 7; ++i) *t += float(std::atof(argv[10 + 3 * i + v[i]]));
    ++calls;
    return ORI_OK;
  };
  float best = 0;
  time(s, &best);
  if (search_schedule(&s, &best, mixed, std::atoi(argv[2]), time) != ORI_OK) return 1;
  for (int i = 0; i < 7; ++i) std::printf("%%d ", *f[i]);
  std::printf("%%d\n", calls);
}
"""


@pytest.fixture(scope="module")
def search(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("no g++")
    with open(os.path.join(ROOT, "paper_1602_04691_gb300", "csrc", "ori_api.cu")) as f:
        src = f.read()
    fn = re.search(r"template <class Time>\nstatic ori_status search_schedule\(.*?\n\}\n", src, re.S)
    assert fn, "the search is a function of its own"
    d = tmp_path_factory.mktemp("search")
    (d / "s.cpp").write_text(MAIN % fn.group(0))
    subprocess.run(["g++", "-std=c++17", "-I" + os.path.join(ROOT, "include"), "-o", str(d / "s"), str(d / "s.cpp")],
                   check=True)

    def run(mixed, nv, start, costs):
        args = [str(int(mixed)), str(nv), *map(str, start), *[str(c) for row in costs for c in row]]
        out = subprocess.run([str(d / "s"), *args], check=True, capture_output=True, text=True).stdout.split()
        return list(map(int, out[:7])), int(out[7])
    return run


@pytest.mark.parametrize("cheap", [0, 1, 2])
def test_every_variant_and_cap_can_win_from_every_start(search, cheap):
    costs = [[1, 2, 9]] * 3 + [[abs(v - cheap) + (0.5 if v > cheap else 0) for v in range(3)]] * 4
    for start_v, start_cap in itertools.product(range(3), range(3)):
        best, calls = search(False, 3, [0, 0, 0] + [start_v] * 3 + [start_cap], costs)
        assert best == [0, 0, 0, cheap, cheap, cheap, cheap], (start_v, start_cap)
        assert calls == 1 + 3 + 3 * 2 + 2


def test_kernel_choices_are_tried_both_ways(search):
    persistent = [[1, 5, 9]] * 3 + [[0, 1, 1]] * 4
    tiles = [[5, 1, 9]] * 3 + [[0, 1, 1]] * 4
    for start in ([0, 0, 0], [1, 1, 1], [1, 0, 1]):
        assert search(False, 3, start + [0] * 4, persistent)[0][:3] == [0, 0, 0]
        assert search(False, 3, start + [0] * 4, tiles)[0][:3] == [1, 1, 1]


def test_a_mixed_length_searches_its_staging_and_the_cap(search):
    costs = [[5, 1, 9]] * 3 + [[9, 8, 1]] + [[2, 1, 0]] + [[9, 8, 1]] + [[1, 2, 3]]
    best, calls = search(True, 2, [0] * 6 + [1], costs)      # a plan given a cap of one gets rid of it
    assert best == [0, 0, 0, 0, 1, 0, 0] and calls == 1 + 1 + 2
