"""Accumulation chunks of one to three K stages (TN_SPLIT_CHUNK): a contracted index
of two or more stages is then several chunks, each an item of its own where the
tiles are few.  Pairs: every tile width of the rule, one tile and several, K from
one stage on; the entry point with static scratch chains the same chunks, so its
output must be equal bit for bit, and FP64 bounds it (split products, 2e-5 as in
the pairwise tests).  Amplitudes: the widest tiles, from a tuner file; every width
adds the same chunks in the same order, so the amplitudes are those of the rule's
own width.  And a pipeline wait that expires in that form."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

PAIRS = """
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

# the 4x5 circuit, depth 1+10+1, 6 open qubits: two steps of log2 M, N, K = (8, 7, 7), one unit each
WIDE = """
import os
import numpy as np
import tn_inputs as I
from _lib import tnlib
T = tnlib()
net = T.build_network(T.random_circuit(4, 5, 10, 1), list(range(14, 20)))
words = I.bitstrings(20, 1, 3)
plans = [T.plan(net, num_sliced=0, search_trials=4, seed=1) for _ in range(2)]
info = plans[0].info()
tensors, _ = plans[0].layout()
shapes = [(t["log2_m"], t["log2_n"], t["log2_k"]) for t in tensors[info["num_leaves"]:]]
assert (8, 7, 7) in shapes, shapes
for precision in ("split_bf16", "split_fp16"):
    with open(os.environ["TN_AUTOTUNE_CACHE"], "a") as f:
        for s, (m, n, k) in enumerate(shapes):
            if m >= 7 and n >= 6 and k >= 3:
                print("%x %d %d %d 8 1" % (info["hash"], T.PREC[precision], s, 128 if n >= 7 else 64), file=f)
for precision in ("split_bf16", "split_fp16"):
    ref = plans[0].contract_amplitudes(words, precision=precision, handover=2)
    got = plans[1].contract_amplitudes(words, precision=precision, handover=2, autotune=True)
    assert np.array_equal(got, ref), precision
"""


def _child(code, **env):
    here = os.path.dirname(os.path.abspath(__file__))
    env = dict(os.environ, PYTHONPATH=os.pathsep.join([here, os.path.dirname(here), os.environ.get("PYTHONPATH", "")]),
               **env)
    r = subprocess.run([sys.executable, "-c", code], env=env, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr


@pytest.mark.parametrize("chunk", [1, 2, 3])
def test_pairs(chunk):
    _child(PAIRS, TN_SPLIT_CHUNK=str(chunk))


@pytest.mark.parametrize("chunk", [1, 2])
def test_wide_tiles_from_a_tuner_file(chunk, tmp_path):
    _child(WIDE, TN_SPLIT_CHUNK=str(chunk), TN_AUTOTUNE_CACHE=str(tmp_path / "tuned"))


def test_expired_wait_with_chunks_as_items_then_the_call_is_correct():
    """One tile whose 16 chunks are items: every pipeline wait gives up at once, and
    the pass that adds the chunks' sums still runs."""
    import torch

    from _lib import tnlib
    from test_gpu_direct import _case
    T = tnlib()
    la, lb, lc, A, B, C, ref, at = _case(7, 7, 13, "random", 0, 11)
    try:
        T.set_wait_limit(0)
        with pytest.raises(T.TnError) as ei:
            T.contract_pair(A, la, B, lb, C, lc, precision="split_bf16", algo="fused_tc")
        assert ei.value.status == 5, ei.value
    finally:
        T.set_wait_limit(-1)
    torch.cuda.synchronize()
    T.contract_pair(A, la, B, lb, C, lc, precision="split_bf16", algo="fused_tc")
    assert float((C[at] - ref).norm()) <= 2e-5 * float(ref.norm())
