"""The tensor-core GEMM that converts its large operand itself (one unit, N <=
64, M >= 2^14, K >= 2^7): every column width, one and several accumulation
chunks, single and several tiles per CTA, each precision, random index orders
and the planner's, operands and output off a 16-byte boundary, against FP64; and
a pipeline wait that expires."""
import pytest

from _lib import tnlib

pytestmark = pytest.mark.gpu
# the bounds of the pairwise tests: split products 2e-5, one 16-bit product 2e-3 (fp16) and 1.5e-2 (bf16)
BOUND = {"split_bf16": 2e-5, "split_fp16": 2e-5, "scaled_fp16": 2e-3, "scaled_bf16": 1.5e-2}


def _case(nm, nn, nk, order, odd, seed):
    import numpy as np
    import torch
    rng = np.random.default_rng(seed)
    x = list(range(nm + nn + nk))
    M, N, K = x[:nm], x[nm:nm + nn], x[nm + nn:]
    la, lb, lc = M + K, N + K, M + N
    if order == "random":
        la, lb, lc = ([int(v) for v in rng.permutation(s)] for s in (la, lb, lc))
    g = torch.Generator(device="cuda").manual_seed(seed)
    A = torch.randn((1 << len(la)) + odd, dtype=torch.complex64, device="cuda", generator=g)[odd:]
    B = torch.randn((1 << len(lb)) + odd, dtype=torch.complex64, device="cuda", generator=g)[odd:]
    C = torch.full(((1 << len(lc)) + odd,), float("nan"), dtype=torch.complex64, device="cuda")[odd:]

    def offsets(ls, group):
        o = torch.zeros(1, dtype=torch.int64, device="cuda")
        for l in group:
            o = (o[:, None] + torch.tensor([0, 1 << (len(ls) - 1 - ls.index(l))], device="cuda")[None, :]).reshape(-1)
        return o

    ref = (A[offsets(la, M)[:, None] + offsets(la, K)[None, :]].to(torch.complex128) @
           B[offsets(lb, K)[:, None] + offsets(lb, N)[None, :]].to(torch.complex128))
    return la, lb, lc, A, B, C, ref, offsets(lc, M)[:, None] + offsets(lc, N)[None, :]


@pytest.mark.parametrize("precision", list(BOUND))
@pytest.mark.parametrize("order", ["random", "planner"])
@pytest.mark.parametrize("nm,nn,nk", [(14, 6, 7), (14, 4, 8), (14, 5, 9), (15, 6, 10), (14, 4, 11), (16, 5, 7)])
def test_matches_fp64(nm, nn, nk, order, precision):
    T = tnlib()
    for odd in (0, 1):
        la, lb, lc, A, B, C, ref, at = _case(nm, nn, nk, order, odd, 100 * nm + 10 * nn + nk + odd)
        T.contract_pair(A, la, B, lb, C, lc, precision=precision, algo="fused_tc")
        assert float((C[at] - ref).norm()) <= BOUND[precision] * float(ref.norm())


def test_expired_wait_returns_etimeout_then_the_call_is_correct():
    T = tnlib()
    la, lb, lc, A, B, C, ref, at = _case(15, 6, 9, "random", 0, 5)
    try:
        T.set_wait_limit(0)
        with pytest.raises(T.TnError) as ei:
            T.contract_pair(A, la, B, lb, C, lc, precision="split_bf16", algo="fused_tc")
        assert ei.value.status == 5, ei.value
    finally:
        T.set_wait_limit(-1)
    T.contract_pair(A, la, B, lb, C, lc, precision="split_bf16", algo="fused_tc")
    assert float((C[at] - ref).norm()) <= 2e-5 * float(ref.norm())
