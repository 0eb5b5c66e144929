"""The linker's totals when a buffer is too small: a total that was never
counted (whatever its memory holds) sizes no scan. The rule is host code too,
and is compiled and run here without a GPU."""
import os
import subprocess

import pytest

from paper_2106_15789_gb300 import build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include "sc_internal.h"
int main(int argc, char** argv) {
  int n[3] = {atoi(argv[1]), atoi(argv[2]), 0};
  const sc::LinkTotals t{n, atoll(argv[3]), atoll(argv[4])};
  printf("%lld %lld %lld %d %d\n", t.scan_length(sc::LINK_SCAN_LEN, 1, 77), t.scan_length(sc::LINK_SCAN_RUNS, 4096, 0),
         t.scan_length(sc::LINK_SCAN_COMPS, 1, 0), t.runs_fit() ? 1 : 0, t.all_fit() ? 1 : 0);
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    d = tmp_path_factory.mktemp("totals")
    (d / "totals.cu").write_text(PROGRAM)
    subprocess.run([build.nvcc(), *build.ARCH, "-std=c++17", "-I", os.path.join(ROOT, "include"), "-I", build.CSRC,
                    str(d / "totals.cu"), "-o", str(d / "totals")], check=True)
    return str(d / "totals")


MAX_RUNS, MAX_COMP = 70000, 9000


@pytest.mark.parametrize("runs", [0, 1, 4096, 4097, MAX_RUNS, MAX_RUNS + 1, 2**31 - 1, -1])
@pytest.mark.parametrize("comps", [0, 5, MAX_COMP, MAX_COMP + 1, 2**31 - 1, -1, -252645136, -(2**31)])
def test_scan_lengths(program, runs, comps):
    out = subprocess.run([program, str(runs), str(comps), str(MAX_RUNS), str(MAX_COMP)], check=True,
                         capture_output=True, text=True).stdout.split()
    of_len, of_runs, of_comps, runs_fit, all_fit = map(int, out)
    assert of_len == 77
    assert runs_fit == (0 <= runs <= MAX_RUNS)
    assert of_runs == (-(-runs // 4096) if runs_fit else -1)
    assert all_fit == (runs_fit and 0 <= comps <= MAX_COMP)
    assert of_comps == (comps if all_fit else -1)  # never past the room, never below -1
