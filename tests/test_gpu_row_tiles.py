"""Streaming contraction by row tiles (2^19 rows and more): every N and K it
takes at the ends of its range, random index orders and the planner's, operands
and output off a 16-byte boundary; against FP64, and bit for bit against the
thread-per-row kernels, which contract the same tensors in two halves."""
import numpy as np
import pytest

from _lib import tnlib

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("order", ["random", "planner"])
@pytest.mark.parametrize("nn,nk", [(0, 2), (2, 0), (1, 1), (4, 0), (0, 4), (4, 1), (2, 3), (3, 4), (4, 4)])
def test_row_tiles_match_fp64_and_the_thread_per_row_kernels(nn, nk, order):
    T = tnlib()
    import torch
    nm = 19
    rng = np.random.default_rng(100 * nn + nk)
    x = list(range(nm + nn + nk))
    M, N, K = x[:nm], x[nm:nm + nn], x[nm + nn:]
    top = M[0]  # slowest in A and C, so halves of both are contiguous
    la, lb, lc = M[1:] + K, N + K, M[1:] + N
    if order == "random":
        la, lb, lc = ([int(v) for v in rng.permutation(s)] for s in (la, lb, lc))
    for odd in (0, 1):
        g = torch.Generator(device="cuda").manual_seed(17 + odd)
        A = torch.randn((1 << (nm + nk)) + odd, dtype=torch.complex64, device="cuda", generator=g)[odd:]
        B = torch.randn((1 << (nn + nk)) + odd, dtype=torch.complex64, device="cuda", generator=g)[odd:]
        C = torch.full(((1 << (nm + nn)) + odd,), float("nan"), dtype=torch.complex64, device="cuda")[odd:]
        T.contract_pair(A, [top] + la, B, lb, C, [top] + lc)
        halves = torch.empty_like(C)
        for h in (0, 1):
            a, c = A.view(2, -1)[h], halves.view(2, -1)[h]
            T.contract_pair(a, la, B, lb, c, lc)
        assert torch.equal(torch.view_as_real(C), torch.view_as_real(halves))
        # FP64 by index arithmetic: rows x K against K x N
        def offsets(ls, group):
            o = torch.zeros(1, dtype=torch.int64, device="cuda")
            for l in group:
                o = (o[:, None] + torch.tensor([0, 1 << (len(ls) - 1 - ls.index(l))], device="cuda")[None, :]).reshape(-1)
            return o
        am, ak = offsets([top] + la, M), offsets([top] + la, K)
        bk, bn = offsets(lb, K), offsets(lb, N)
        cm, cn = offsets([top] + lc, M), offsets([top] + lc, N)
        ref = A[am[:, None] + ak[None, :]].to(torch.complex128) @ B[bk[:, None] + bn[None, :]].to(torch.complex128)
        got = C[cm[:, None] + cn[None, :]].to(torch.complex128)
        # at most 16 products in FP32: a few 2^-24 of the sum's size
        assert float((got - ref).norm()) <= 1e-6 * float(ref.norm())
