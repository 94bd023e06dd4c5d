"""The fused digit-plane product (every digit pair of a tile in one kernel) through the C ABI.

Integers of at most 18 bits need four base-64 digits, so no digit pair within the kept levels is cut off and
the result (below 2^53) has to be the exact integer, whatever the tiling: row and column remainders,
operands that change places, K split over blocks, K long enough for several drains of the level
accumulators (2048 of K each at level 9), and one tile or many per block.
"""
import numpy as np
import pytest

from paper_2010_04768_gb300 import gfcc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,N,K", [(1, 1, 1), (128, 64, 64), (127, 33, 65), (40, 300, 9000), (300, 40, 9000),
                                   (5000, 70, 130), (640, 1300, 2300), (200, 16, 70000)])
def test_integer_products_are_exact(M, N, K):
    rng = np.random.default_rng(M + 3 * N + 7 * K)
    A = rng.integers(-(1 << 17), 1 << 17, size=(M, K)).astype(np.float64)
    B = rng.integers(-(1 << 17), 1 << 17, size=(N, K)).astype(np.float64)
    A[:, 0] = 1 << 17                                # the largest digits in one column
    B[:, 0] = -(1 << 17)
    ref = np.rint(A @ B.T)
    assert np.abs(ref).max() < 2.0**53
    big = np.abs(A[:4]) @ np.abs(B[:4]).T < 2.0**53  # every partial sum is exact in the reference too
    assert big.all()
    assert np.array_equal(gfcc.selftest_gemm_f64emu(A, B, S=8, P=9), ref)


@pytest.mark.parametrize("S,P", [(1, 2), (2, 3), (3, 4), (4, 5), (5, 6), (6, 7), (7, 8), (8, 8), (8, 9)])
def test_every_level(S, P):
    # a term is cut at 2^-(6P - 4) of the product of its row scales (at most twice the largest magnitudes)
    rng = np.random.default_rng(S)
    M, N, K = 150, 90, 3000
    A, B = rng.standard_normal((M, K)), rng.standard_normal((N, K))
    bound = 2.0 ** (4 - 6 * P) * K * 4 * np.abs(A).max(1)[:, None] * 4 * np.abs(B).max(1)[None, :]
    C = gfcc.selftest_gemm_f64emu(A, B, S=S, P=P)
    assert np.all(np.abs(C - A @ B.T) <= bound + 1e-13 * np.abs(A) @ np.abs(B).T)
