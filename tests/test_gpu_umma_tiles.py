"""BF16 products over CTA pairs at each tile width (chosen by the waves of 76 pairs) and the row-wise stores of every
kernel, at rows that do not align to 16 bytes and columns past the last full block."""
import numpy as np
import pytest

from paper_2010_04768_gb300 import gfcc

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="session", autouse=True)
def _built():
    from paper_2010_04768_gb300 import build
    build.build()
    gfcc.load()


def check(M, N, K):
    rng = np.random.default_rng(M + N + K)
    A = rng.integers(-8, 9, (M, K)).astype(np.float32)
    B = rng.integers(-8, 9, (N, K)).astype(np.float32)
    # integers: every sum of products below 64 K <= 2^24 is exact in FP32
    assert 64 * K <= 2 ** 24
    assert np.array_equal(gfcc.selftest_gemm_bf16(A, B), A @ B.T)


# 128 columns (one wave), 192 (128 would need a second), 256 (192 would)
@pytest.mark.parametrize("M,N,K", [(300, 132, 520), (600, 4000, 520), (530, 4001, 530), (600, 5000, 520), (515, 4999, 521)])
def test_pair_widths(M, N, K):
    gfcc.set_process_option(gfcc.OPT_GEMM_PAIR, 1.0)
    try:
        check(M, N, K)
    finally:
        gfcc.set_process_option(gfcc.OPT_GEMM_PAIR, 0.0)


@pytest.mark.parametrize("persist", [1.0, 2.0])
@pytest.mark.parametrize("M,N,K", [(40000, 60, 133), (129, 33, 64), (200, 30, 70), (260, 255, 129), (127, 1, 200)])
def test_row_stores(persist, M, N, K):
    gfcc.set_process_option(gfcc.OPT_GEMM_PERSIST, persist)
    try:
        check(M, N, K)
    finally:
        gfcc.set_process_option(gfcc.OPT_GEMM_PERSIST, 0.0)
