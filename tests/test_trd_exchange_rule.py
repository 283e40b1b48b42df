"""The meeting counter of the resident reduction (csrc/tdc_trd_rule.cuh), stepped through on
the CPU for every order the kernel takes and grids below, at and above it: at each step exactly
the blocks that the target counts arrive, the owner of the exchanged column is one of them, and
the step's results are written by a block that is still there."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
RULE = os.path.join(ROOT, "paper_2008_01990_gb300", "csrc", "tdc_trd_rule.cuh")

# k_trd_resident's control flow: a block returns at once unless it takes part in step 0
# (argument 3 = 1: only blocks beyond the order do, so that the owner of column 0 alone arrives
# uncounted); at step k it arrives, and leaves unless it takes part in step k + 1.
PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include "%s"
using namespace tdc;
int main(int argc, char** argv) {
  const int G = atoi(argv[1]), top = atoi(argv[2]), all_enter = atoi(argv[3]);
  static int last[4096];
  for (int m = 3; m <= top; ++m) {
    const int nb = m < G ? m : G;
    static bool in[4096];
    for (int b = 0; b < nb; ++b) {
      last[b] = trd_res_last(b, m, G);
      if (last[b] >= m || last[b] + G < m || last[b] %% G != b) { printf("m %%d: last column of %%d\n", m, b); return 1; }
      in[b] = all_enter || trd_res_takes_part(last[b], 0);
    }
    long long counter = 0, target = 0;
    for (int k = 0; k + 2 < m; ++k) {
      target += trd_res_arrivals(k, m, G);
      if (!in[(k + 1) %% G]) { printf("m %%d step %%d: the owner of column k + 1 is gone\n", m, k); return 1; }
      for (int b = 0; b < nb; ++b) {
        if (!in[b]) continue;
        ++counter;
        if (!trd_res_takes_part(last[b], k + 1)) in[b] = false;
      }
      if (counter != target) { printf("m %%d step %%d: %%lld arrivals, target %%lld\n", m, k, counter, target); return 2; }
      const int w = trd_res_writer(k, m, G);
      if (w < 0 || w >= nb || !in[w]) { printf("m %%d step %%d: the writer is gone\n", m, k); return 1; }
    }
    for (int b = 0; b < nb; ++b)
      if (in[b] != (b == (m - 1) %% G)) { printf("m %%d: block %%d at the end\n", m, b); return 1; }
  }
  return 0;
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    d = tmp_path_factory.mktemp("trd_rule")
    src, exe = d / "rule.cpp", d / "rule"
    src.write_text(PROGRAM % RULE)
    subprocess.run(["g++", "-O2", "-std=c++17", "-o", str(exe), str(src)], check=True)
    return str(exe)


@pytest.mark.parametrize("G", [1, 2, 3, 7, 64, 148, 152, 160, 2000])
def test_arrivals_are_those_the_target_counts(program, G):
    r = subprocess.run([program, str(G), "1824" if G >= 148 else "600", "0"], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout


@pytest.mark.parametrize("G", [3, 148, 152])
def test_an_uncounted_arrival_is_found(program, G):
    """The same steps with every block entering: for m <= G the owner of column 0 arrives
    without being counted, and the walk says so."""
    r = subprocess.run([program, str(G), str(G), "1"], capture_output=True, text=True)
    assert r.returncode == 2 and "m 3 step 0" in r.stdout, r.stdout
