"""Operand split pass and output order of the tensor-core contraction: random
index orders of all three tensors at the edges of the pass's tiles (the
smallest operands, 2^9, 2^10, 2^12 elements and around the switch to large
tiles), every precision, and operands that start off a 16-byte boundary."""
import numpy as np
import pytest

from _lib import tnlib

pytestmark = pytest.mark.gpu
LETTERS = "abcdefghijklmnopqrstuvwxyzABCDEFGHIJKLMNOPQRSTUVWXYZ"
# the bounds of the pairwise tests: split products 2e-5, one 16-bit product 2e-3 (fp16) and 1.5e-2 (bf16)
BOUND = {"split_bf16": 2e-5, "split_fp16": 2e-5, "scaled_fp16": 2e-3, "scaled_bf16": 1.5e-2}


@pytest.mark.parametrize("precision", list(BOUND))
@pytest.mark.parametrize("nm,nn,nk", [(7, 4, 3), (7, 6, 3), (8, 4, 5), (9, 5, 3), (7, 7, 5), (12, 4, 8), (11, 7, 10),
                                      (16, 4, 6)])
def test_random_orders_match_fp64(nm, nn, nk, precision):
    T = tnlib()
    import torch
    rng = np.random.default_rng(1000 * nm + 100 * nn + nk)
    x = list(range(nm + nn + nk))
    M, N, K = x[:nm], x[nm:nm + nn], x[nm + nn:]
    sub = lambda ls: "".join(LETTERS[v] for v in ls)
    for odd in (0, 1):
        la, lb, lc = ([int(v) for v in rng.permutation(s)] for s in (M + K, N + K, M + N))
        g = torch.Generator(device="cuda").manual_seed(7 + odd)
        # odd: one element past an aligned base (8-byte alignment only)
        A = torch.randn((1 << len(la)) + odd, dtype=torch.complex64, device="cuda", generator=g)[odd:]
        B = torch.randn((1 << len(lb)) + odd, dtype=torch.complex64, device="cuda", generator=g)[odd:]
        C = torch.full(((1 << len(lc)) + odd,), float("nan"), dtype=torch.complex64, device="cuda")[odd:]
        ref = np.einsum(f"{sub(la)},{sub(lb)}->{sub(lc)}", A.cpu().numpy().astype(np.complex128).reshape((2,) * len(la)),
                        B.cpu().numpy().astype(np.complex128).reshape((2,) * len(lb)), optimize=True).reshape(-1)
        T.contract_pair(A, la, B, lb, C, lc, precision=precision, algo="fused_tc")
        got = C.cpu().numpy().astype(np.complex128)
        assert np.linalg.norm(got - ref) <= BOUND[precision] * np.linalg.norm(ref), (odd, la, lb, lc)
