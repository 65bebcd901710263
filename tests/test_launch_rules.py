"""Host rules of the kernels' launches, compiled alone from the library's
headers and checked without a GPU."""
import os
import subprocess

import pytest

from conftest import ROOT

CSRC = os.path.join(ROOT, "paper_1301_5887_gb300", "csrc")


def _run(tmp_path, body):
    src = tmp_path / "rule.cu"
    src.write_text('#include <cstdio>\n#include "internal.h"\n#include "runtime.h"\nusing namespace wedge;\n'
                   "int main() {\n%s\n}\n" % body)
    exe = tmp_path / "rule"
    subprocess.run(["nvcc", "-std=c++17", "-I", CSRC, "-o", str(exe), str(src)], check=True)
    return subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout.split()


@pytest.mark.parametrize("ready,first", [("unused", 1), ("cleared", 1), ("histograms", 0)])
def test_sort_pass_waits_for_the_clear_of_its_tickets(tmp_path, ready, first):
    """A chained pass takes tickets before it waits for the operation before it, so that
    operation is never their clear: with the histograms ready it is, for pass 0."""
    out = _run(tmp_path, """
  for (int64_t tiles : {int64_t(1), int64_t(152), CHAIN_TILES, CHAIN_TILES + 1})
    for (int p = 0; p < SORT_MAX_PASSES; ++p)
      printf("%%d ", (int)sort_pass_chained(SortScratch::%s, p, tiles));""" % ready)
    few = [first] + [1] * 7
    assert [int(x) for x in out] == few * 3 + [0] * 8


def test_once_per_device(tmp_path):
    """What a kernel needs before its first launch is done on each device, and again where it failed."""
    out = _run(tmp_path, """
  OncePerDevice once;
  int runs[3] = {};
  auto on = [&](int dev, wedge_status st) {
    once.on(dev, [&] { ++runs[dev]; return st; });
  };
  on(0, WEDGE_ECUDA);
  on(0, WEDGE_OK);
  on(0, WEDGE_OK);
  on(2, WEDGE_OK);
  on(1, WEDGE_OK);
  on(2, WEDGE_ECUDA);
  printf("%d %d %d", runs[0], runs[1], runs[2]);""")
    assert [int(x) for x in out] == [2, 1, 1]
