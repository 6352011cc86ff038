"""The autotuner times the tile widths that the rule weighs, so it finds the rule's
own choice at every shape and number of units."""
from _cxx import run_cxx

PROGRAM = """
#include <cstdio>
#include "kernels.h"
int main() {
  int bad = 0, narrow = 0;
  for (int nm = 7; nm <= 26; ++nm)
    for (int nn = 4; nm + nn <= 30; ++nn)
      for (int units : {1, 2, 5, 16, 150, 1024}) {
        tn::GemmDesc d{};
        d.nm = nm;
        d.nn = nn;
        d.nk = 4;
        d.units = d.units_lo = units;
        int w[3];
        const int n = tn::tma_tile_widths(d, w), rule = tn::tma_tile_n(d);
        bool found = false;
        for (int i = 0; i < n; ++i) {
          found |= w[i] == rule;
          tn::GemmDesc t = d;  // and a width it finds is one that the launch takes
          t.tile_n = w[i];
          if (tn::tma_tile_n(t) != w[i]) ++bad;
        }
        narrow += rule == 32 && nn > 5;
        if (!found) {
          std::printf("M = 2^%d, N = 2^%d, %d units: %d columns\\n", nm, nn, units, rule);
          ++bad;
        }
      }
  return bad != 0 || narrow == 0;
}
"""


def test_the_rules_width_is_among_those_timed(tmp_path):
    run_cxx(tmp_path, PROGRAM)


def test_the_tuner_takes_its_widths_from_the_rule():
    import os

    from paper_2110_14502_gb300 import build as B
    with open(os.path.join(B.CSRC, "executor.cu")) as f:
        text = f.read()
    tuner = text[text.index("c.tuning) {"):text.index("E.tuned.push_back({c.precision")]
    assert "tma_tile_widths(d, widths)" in tuner, tuner
