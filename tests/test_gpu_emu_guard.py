"""The digit planes that take the place of FP64 contractions: error bound of FP64 sums for rows of any spread, infinities
and NaN as FP64 gives them, and exact sums of the largest digits at the edges of the K blocks."""
import numpy as np
import pytest

from paper_2010_04768_gb300 import gfcc

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2010_04768_gb300 import build
    build.build()
    gfcc.load()


def rows(rng, kind, n, K):
    X = rng.standard_normal((n, K))
    if kind == "spread":                 # magnitudes even over 2^40
        X = np.sign(X) * 2.0 ** (-40 * rng.random((n, K)))
    elif kind == "crossed":              # the large entries of one operand meet the small ones of the other
        X = X * 2.0 ** (-40.0 * (np.arange(K) < K // 2))
    elif kind == "spike":                # one large entry, the others 2^-40 of it
        X = X * 2.0 ** -40
        X[np.arange(n), rng.integers(0, K, n)] = 1.0
    elif kind == "decay":                # Cholesky vectors
        X = X * np.exp(-np.arange(K) / 12.0)
    elif kind == "sparse":               # products of zeros
        X = X * (rng.random((n, K)) < 0.05)
    return X


def beyond(C, A, B, C0):
    """Outputs further from the exact values than K 2^-53 times the sum of magnitudes (and the rounding of C0)."""
    L = np.longdouble
    ref = A.astype(L) @ B.T.astype(L) + C0
    bound = (A.shape[1] + 2) * 2.0 ** -53 * (np.abs(A) @ np.abs(B).T + np.abs(C0))
    return np.abs(C - ref) > bound


@pytest.mark.parametrize("K", [33, 64, 200, 384, 385, 700])
@pytest.mark.parametrize("kind", ["gauss", "spread", "crossed", "spike", "decay", "sparse"])
def test_outputs_hold_the_fp64_bound(kind, K):
    rng = np.random.default_rng(K)
    M, N = 131, 77
    A, B = rows(rng, kind, M, K), rows(rng, kind, N, K)
    if kind == "crossed":
        B = B[:, ::-1].copy()
    C0 = rng.standard_normal((M, N)) * 2.0 ** -30
    for mode in (1, 2):
        assert not beyond(gfcc.selftest_gemm_planes(A, B, mode), A, B, 0.0).any()
        assert not beyond(gfcc.selftest_gemm_planes(A, B, mode, C0), A, B, C0).any()
    if kind in ("crossed", "spike"):     # what the planes alone give
        assert beyond(gfcc.selftest_gemm_planes(A, B, 0), A, B, 0.0).any()


def test_few_small_outputs_among_many():
    # single outputs in FP64, the others from the planes: long sums (K split) and short ones, both orders of M and N
    rng = np.random.default_rng(5)
    for M, N, K in ((300, 500, 96), (20, 40, 40000), (700, 9, 5000)):
        A, B = rng.standard_normal((M, K)), rng.standard_normal((N, K))
        A[3, 1:] *= 2.0 ** -40           # row 3 against column 5: 2^-40 each
        A[3, 0] = B[5, 1] = 1.0
        B[5, 2:] *= 2.0 ** -40
        B[5, 0] = 2.0 ** -40
        for mode in (1, 2):
            assert not beyond(gfcc.selftest_gemm_planes(A, B, mode), A, B, 0.0).any()
        assert beyond(gfcc.selftest_gemm_planes(A, B, 0), A, B, 0.0).any()


@pytest.mark.parametrize("many", [False, True])
def test_infinities_and_nan(many):
    rng = np.random.default_rng(7)
    A, B = rng.standard_normal((64 if many else 500, 100)), rng.standard_normal((700, 100))
    A[5, 7], A[6, 8], A[7, 9] = np.inf, -np.inf, np.nan
    B[1, 7] = 0.0
    if many:
        A[:, 3] = np.inf
    with np.errstate(invalid="ignore"):
        ref = A @ B.T
    for mode in (1, 2):
        C = gfcc.selftest_gemm_planes(A, B, mode)
        assert np.array_equal(np.isnan(C), np.isnan(ref))
        inf = np.isinf(ref)
        assert np.array_equal(C[inf], ref[inf]) and np.array_equal(np.isinf(C), inf)
        ok = np.isfinite(ref)
        assert np.allclose(C[ok], ref[ok], rtol=0, atol=1e-12)


@pytest.mark.parametrize("K", [1, 63, 64, 383, 384, 385, 512, 513, 1024, 1025])
@pytest.mark.parametrize("rows_", [(33, 65), (129, 31)])
def test_largest_digits_are_summed_exactly(K, rows_):
    # rows of numbers whose first digits are +-128 (sums of at most 384 terms) or +-63 and whose others are +-64 or 63: a
    # level that passed 2^24 would be off by a unit of 2^(-7 level), against the 2^-54 a term that the planes leave out
    rng = np.random.default_rng(K)
    M, N = rows_
    first, cut = (128, 127) if K <= 384 else (63, 62)

    def numbers(n):
        d = rng.choice([-64, 63], size=(n, K, 6))
        lead = rng.choice([first, -cut], size=(n, K)) if n % 2 else np.full((n, K), first)
        d[lead == 128] = -64             # below 1
        Y = lead.astype(object) * 2 ** 42
        for i in range(6):
            Y = Y + d[:, :, i].astype(object) * 2 ** (35 - 7 * i)
        return Y                          # times 2^-49

    YA, YB = numbers(M), numbers(N)
    A, B = YA.astype(np.float64) * 2.0 ** -49, YB.astype(np.float64) * 2.0 ** -49
    C = gfcc.selftest_gemm_planes(A, B, 0)
    exact = YA @ YB.T                     # times 2^-98, Python integers
    err = np.array([[abs(int(c * 2.0 ** 98) - e) for c, e in zip(r, q)] for r, q in zip(C, exact)], dtype=np.float64)
    assert (err <= K * 2.0 ** 44 + np.abs(C) * 2.0 ** 45 + 1).all()
