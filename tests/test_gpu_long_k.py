"""The tensor-core GEMM with a long K and few tiles, whose accumulation chunks run
on SMs of their own: one tile and the most tiles of the rule, two chunks (the
last of its range) and many, every column width, outputs off a 16-byte boundary.
The entry point with static scratch never takes that path and adds the same
chunks in the same order, so its output must be equal bit for bit; FP64 bounds
the scaled format (split products, 2e-5 as in the pairwise tests)."""
import pytest

from _lib import tnlib
from test_gpu_direct import _case

pytestmark = pytest.mark.gpu
SHAPES = [(7, 4, 10), (8, 5, 11), (7, 7, 13), (9, 6, 12), (13, 7, 10), (8, 4, 14), (10, 9, 10)]


@pytest.mark.parametrize("order", ["random", "planner"])
@pytest.mark.parametrize("nm,nn,nk", SHAPES)
def test_same_bits_as_without_the_space_for_sums(nm, nn, nk, order):
    T = tnlib()
    import torch
    for odd in (0, 1):
        la, lb, lc, A, B, C, ref, at = _case(nm, nn, nk, order, odd, 100 * nm + 10 * nn + nk + odd)
        T.contract_pair(A, la, B, lb, C, lc, precision="split_bf16", algo="fused_tc")
        assert float((C[at] - ref).norm()) <= 2e-5 * float(ref.norm())
        if 8 * (2**nm + 2**nn) * 2**nk <= 64 << 20:  # the static array's size
            D = torch.full_like(C, float("nan"))
            T.contract_pair_noalloc(A, la, B, lb, D, lc)
            torch.cuda.synchronize()
            assert torch.equal(torch.view_as_real(C), torch.view_as_real(D))


@pytest.mark.parametrize("nm,nn,nk", SHAPES)
def test_split_fp16_matches_fp64(nm, nn, nk):
    T = tnlib()
    la, lb, lc, A, B, C, ref, at = _case(nm, nn, nk, "random", 1, nm + nn + nk)
    A *= 2.0**70  # exponents beyond one factor's range are applied to the sum
    T.contract_pair(A, la, B, lb, C, lc, precision="split_fp16", algo="fused_tc")
    assert float((C[at] / 2.0**70 - ref).norm()) <= 2e-5 * float(ref.norm())
