"""The default kernels' choice between full tiles and tiles of two elements, on the host.

The rule is compiled from its header for every number of points and run for every slot count up to
20000 on 152 multiprocessors.  Whatever margin it keeps, it has to take the small tiles where full ones
of the kernel's own width leave half of the multiprocessors without a tile and small ones would halve
the work of the fullest, and must not take them where they save less than an eighth.
"""
import subprocess

import pytest

from paper_2512_08571_gb300 import build as B

SRC = r"""
#include <cstdio>
#include "fe_ks_line_ff.cuh"
using namespace feks;
static int64_t most(int64_t slots, int vg) { return ((slots + vg - 1) / vg + 151) / 152 * vg; }
static int bad = 0;
static void check(const char* kernel, int nq, int vg, int64_t slots, bool small) {
  const int64_t full = most(slots, vg), two = most(slots, 2);
  const bool must = 2 * ((slots + vg - 1) / vg) <= 152 && 2 * two <= full, may = 8 * two <= 7 * full;
  if ((must && !small) || (small && !may)) {
    if (bad++ < 20) printf("%s n_q %d slots %lld small %d\n", kernel, nq, (long long)slots, (int)small);
  }
}
template <int NQ>
static void run() {
  for (int64_t s = 1; s <= 20000; ++s) {
    if constexpr (line_vg(NQ, false) > 2)
      check("line", NQ, line_vg(NQ, false), s, line_small<line_vg(NQ, false), line_vg(NQ, true)>(s, 152));
    if constexpr (line_ff_vg(NQ, false) > 2) check("pairs", NQ, line_ff_vg(NQ, false), s, line_ff_small<NQ>(s, 152));
  }
}
int main() {
  run<2>(), run<3>(), run<4>(), run<5>(), run<6>(), run<7>(), run<8>(), run<9>(), run<10>(), run<11>();
  return bad != 0;
}
"""


def test_small_tiles_where_full_ones_leave_multiprocessors_idle(tmp_path):
    try:
        nvcc = B._nvcc()
    except RuntimeError:
        pytest.skip("no nvcc")
    (tmp_path / "rule.cu").write_text(SRC)
    exe = tmp_path / "rule"
    r = subprocess.run([nvcc, *B.ARCH, *B.FLAGS, "-I" + B.CSRC, str(tmp_path / "rule.cu"), "-o", str(exe)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
