"""FP32 GEMM steps with many more columns than rows: the tile's columns go to
grid.y, whose limit the tile choice has to keep to."""
import numpy as np
import pytest

from _cxx import run_cxx
from _lib import tnlib

# every M, and N up to 2^22: 128-column tiles fit grid.y there
EVERY_SHAPE = """
#include <cstdio>
#include "kernels.h"
int main() {
  int bad = 0;
  for (int nm = 0; nm <= 30; ++nm)
    for (int nn = 0; nn <= 22; ++nn)
      for (int units : {1, 7, 152, 4096}) {
        tn::GemmDesc d{};
        d.nm = nm;
        d.nn = nn;
        d.units = units;
        const tn::SimtTile t = tn::simt_tile(d);
        if (((int64_t(1) << nn) + t.cols - 1) / t.cols > 65535) {
          std::printf("M = 2^%d, N = 2^%d, %d units: %d columns per tile\\n", nm, nn, units, t.cols);
          ++bad;
        }
      }
  return bad != 0;
}
"""


def test_every_tile_choice_fits_the_grid(tmp_path):
    run_cxx(tmp_path, EVERY_SHAPE)


@pytest.mark.gpu
@pytest.mark.parametrize("algo", ["auto", "fused_simt"])
@pytest.mark.parametrize("nm,nn,nk", [(3, 21, 0), (2, 21, 3), (0, 22, 1), (5, 22, 3), (6, 20, 2)])
def test_wide_columns_match_fp64(nm, nn, nk, algo):
    """Against FP64, at the error bound of the other complex64 pair tests."""
    import torch
    T = tnlib()
    g = torch.Generator(device="cuda").manual_seed(nm + 100 * nn + nk)
    rand = lambda bits: torch.randn(1 << bits, dtype=torch.complex64, device="cuda", generator=g)
    m, n, k = list(range(nm)), list(range(nm, nm + nn)), list(range(nm + nn, nm + nn + nk))
    A, B = rand(nm + nk), rand(nk + nn)
    C = torch.full((1 << (nm + nn),), float("nan"), dtype=torch.complex64, device="cuda")
    T.contract_pair(A, m + k, B, k + n, C, n + m, algo=algo)
    torch.cuda.synchronize()
    ref = (A.view(1 << nm, 1 << nk).to(torch.complex128) @ B.view(1 << nk, 1 << nn).to(torch.complex128)).T
    err = float((C.view(1 << nn, 1 << nm) - ref).norm() / ref.norm())
    assert err <= 1e-5, err
