"""Reduced models over lists of different length, with odd counts of numbers before the model matrices."""
import numpy as np
import pytest

from paper_2010_04768_gb300 import gfcc
from paper_2010_04768_gb300.synthetic import make_problem

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2010_04768_gb300 import build
    build.build()
    gfcc.load()


@pytest.mark.parametrize("o,v", [(4, 16), (5, 15)])   # 100 and 155 coordinates
def test_rows_and_columns_of_different_count(o, v):
    g = gfcc.GFCC(make_problem(o, v, 30, seed=o), sectors="IP")
    orbs = np.arange(1, 4)
    mor = gfcc.MOR(g, "IP")
    mor.expand([-0.9, -0.4], 0.05, orbs, 1e-10)
    assert mor.dim() == 12
    om = np.linspace(-0.9, -0.4, 9)
    G, rr = mor.green(om, 0.05, orbs, residuals=True)
    for P, Q in (([1, 2, 3], [2, 3]), ([3], [1, 2]), ([1, 3], [2])):   # nb + nl odd, n + m even and odd
        H, r = mor.green(om, 0.05, P, Q, residuals=True)
        rows, cols = np.array(P) - 1, np.array(Q) - 1
        assert np.abs(H - G[:, rows][:, :, cols]).max() <= 1e-12 * np.abs(G).max()
        assert np.abs(r - rr[:, rows]).max() <= 1e-12
    mor.close()
    g.close()


def test_model_beyond_shared_memory():
    # more than 117 vectors: matrix and multipliers in the call's workspace; the model interpolates its samples
    om, orbs, eta = np.linspace(-1.6, 0.2, 16), np.arange(12), 0.05
    g = gfcc.GFCC(make_problem(6, 40, 60, seed=3, t1_std=0.05, t2_std=0.05, chol_sigma=0.1), sectors="IP")
    mor = gfcc.MOR(g, "IP")
    try:
        ref, code = mor.expand(om, eta, orbs, 1e-9)
        assert code == gfcc.OK and mor.dim() > 117
        G = mor.green(om, eta, orbs)
        # the samples' solutions lie in the model's space to 1e-9 of |b|, and |A^-1| <= 1 / eta
        assert np.abs(G - ref).max() <= 1e-6 * np.abs(ref).max()
    finally:
        mor.close()
        g.close()
