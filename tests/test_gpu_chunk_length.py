"""Accumulation chunks of one to three K stages (TN_SPLIT_CHUNK): a contracted index
of two or more stages is then several chunks, each an item of its own where the
tiles are few.  Every tile width, one tile and several, K from one stage on; the entry point with static scratch chains the same chunks, so its output
must be equal bit for bit, and FP64 bounds it (split products, 2e-5 as in the
pairwise tests)."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

CHILD = """
import torch
from _lib import tnlib
from test_gpu_direct import _case
T = tnlib()
for nm, nn, nk in [(7, 4, 6), (8, 5, 7), (7, 6, 5), (7, 6, 6), (9, 6, 7), (7, 7, 6), (8, 7, 7), (9, 8, 7), (7, 7, 9)]:
    for order in ("random", "planner"):
        la, lb, lc, A, B, C, ref, at = _case(nm, nn, nk, order, 0, 10000 + 100 * nm + 10 * nn + nk)
        T.contract_pair(A, la, B, lb, C, lc, precision="split_bf16", algo="fused_tc")
        assert float((C[at] - ref).norm()) <= 2e-5 * float(ref.norm()), (nm, nn, nk, order)
        D = torch.full_like(C, float("nan"))
        T.contract_pair_noalloc(A, la, B, lb, D, lc)
        torch.cuda.synchronize()
        assert torch.equal(torch.view_as_real(C), torch.view_as_real(D)), (nm, nn, nk, order)
"""


@pytest.mark.parametrize("chunk", [1, 2, 3])
def test_short_chunks(chunk):
    here = os.path.dirname(os.path.abspath(__file__))
    env = dict(os.environ, TN_SPLIT_CHUNK=str(chunk),
               PYTHONPATH=os.pathsep.join([here, os.path.dirname(here), os.environ.get("PYTHONPATH", "")]))
    r = subprocess.run([sys.executable, "-c", CHILD], env=env, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr
