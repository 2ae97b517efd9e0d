"""The whole-loop kernel's exchange buffer, on the host: the entries that every
rank of a cluster reads and writes in every pass of H_a and H_a^*, from the
index functions that the kernel itself uses.  Ranks meet only between passes,
so inside a pass no rank may write an entry that another one reads or writes;
and what a pass reads has to be what the pass before it wrote."""
import subprocess

import pytest

from paper_1810_11685_gb300 import build

HARNESS = r"""
#include <cstdio>
#include <cstdlib>
#include <vector>
#include "loop2d.cuh"
using namespace qpat;

static int faults = 0;

template <bool ADJ, bool LL>
void check(int nx, int ny, int nc, int nt) {
  const int P = LL ? 4 : 6, nxh = nx / 2 + 1, pairs = ny / 2;
  const int rp = (pairs + nc - 1) / nc, cp = (nxh + nc - 1) / nc;
  const int g0 = ADJ ? 0 : LL ? -1 : -2, g1 = ADJ ? nt * P - 3 : (nt - 1) * P + (LL ? 0 : 1);
  std::vector<int> last((size_t)ny * nx, -1000);                 // pass that wrote the entry
  for (int g = g0; g < g1; ++g) {
    const LoopStep st = loop_pass<ADJ, LL>(g, nt);
    std::vector<int> rd((size_t)ny * nx, -1), wr((size_t)ny * nx, -1);
    auto fault = [&](const char* what, int rank, LoopCell q) {
      if (faults++ < 10)
        printf("%s nx %d ny %d ranks %d pass %d rank %d entry (%d, %d)\n", what, nx, ny, nc, st.ph, rank, q.row, q.col);
    };
    const bool row = loop_is_row(st.ph);
    for (int rank = 0; rank < nc; ++rank) {
      const int per = row ? rp : cp, all = row ? pairs : nxh, pts = row ? nx : ny;
      for (int line = rank * per; line < all && line < (rank + 1) * per; ++line)
        for (int i = 0; i < pts; ++i) {
          if (!(st.flags & kSkipInput))
            loop_with_in<ADJ>(st.ph, [&](auto kind) {
              for (int w = 0; w < 2; ++w) {
                const LoopCell q = loop_in_cell(decltype(kind)::value, line, i, w, nx);
                const size_t at = (size_t)q.row * nx + q.col;
                if (last[at] != g - 1) fault("stale", rank, q);
                rd[at] = rd[at] == -1 || rd[at] == rank ? rank : -2;
              }
            });
          if (!(st.flags & kSkipOutput))
            loop_with_out<ADJ>(st.ph, [&](auto kind) {
              constexpr int k = decltype(kind)::value;
              const bool two = k == kOutRow2 || (k == kOutCol2 && loop_mirror(line, nx) != line);
              for (int w = 0; w < (two ? 2 : 1); ++w) {
                const LoopCell q = loop_out_cell(k, line, i, w, nx);
                const size_t at = (size_t)q.row * nx + q.col;
                if (wr[at] != -1) fault("two writes", rank, q);
                wr[at] = rank;
              }
            });
        }
    }
    for (int q = 0; q < ny * nx; ++q)
      if (wr[q] != -1) {
        if (rd[q] != -1 && rd[q] != wr[q]) fault("race", wr[q], LoopCell{q / nx, q % nx});
        last[q] = g;
      }
  }
}

int main(int argc, char** argv) {
  for (int k = 1; k + 1 < argc; k += 2)
    for (int nc : {16, 8, 4}) {
      const int nx = atoi(argv[k]), ny = atoi(argv[k + 1]);
      check<false, false>(nx, ny, nc, 4);
      check<false, true>(nx, ny, nc, 4);
      check<true, false>(nx, ny, nc, 4);
      check<true, true>(nx, ny, nc, 4);
    }
  printf("%d faults\n", faults);
  return faults != 0;
}
"""

GRIDS = [(168, 168), (24, 24), (24, 30), (96, 96), (150, 210), (216, 48), (56, 40), (224, 224)]


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    d = tmp_path_factory.mktemp("exchange")
    src, exe = d / "exchange.cu", d / "exchange"
    src.write_text(HARNESS)
    subprocess.run([build.nvcc(), *build.ARCH, *build.FLAGS, str(src), "-o", str(exe)], check=True)
    return str(exe)


@pytest.mark.parametrize("grid", GRIDS)
def test_no_rank_writes_what_another_uses_in_a_pass(harness, grid):
    r = subprocess.run([harness, *map(str, grid)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
