"""The FP64 contraction's tile shapes through the FP64 sigma product, against the CPU oracle.

The vector count sets the column count of the narrow contractions (2 columns per vector), so the
cases reach every tile shape (64 x 4, 32 x 8, 16 x 16, 8 x 32, 4 x 64, 32 x 32), K ranges shared by a
cluster, and K split through global memory (o o v or o v v of at least 8192), with ragged edges.
Tolerance: sums of at most 2^14 products in 64 bits, 2^14 x 2^-53 = 2e-12 relative to the sum of
magnitudes at worst; 1e-12 of the largest element as for the other FP64 parity tests.
"""
import numpy as np
import pytest

from oracle.gfcc_ref import GFCCOracle
from paper_2010_04768_gb300 import gfcc
from paper_2010_04768_gb300.synthetic import make_problem, random_vector

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="session", autouse=True)
def _built():
    from paper_2010_04768_gb300 import build
    build.build()
    gfcc.load()


@pytest.mark.parametrize("o,v,L,nvec", [(1, 2, 3, 1), (2, 3, 5, 2), (4, 12, 20, 1), (4, 12, 20, 64), (5, 33, 40, 3),
                                        (9, 41, 50, 16), (14, 50, 60, 1), (4, 46, 50, 5)])
def test_sigma_over_tile_shapes(o, v, L, nvec):
    pr = make_problem(o, v, L, seed=3 * o + v + nvec, t1_std=0.05, t2_std=0.05, chol_sigma=0.3)
    g = gfcc.GFCC(pr)
    orc = GFCCOracle(pr.fock, pr.chol, pr.t1, pr.t2, o=o)
    for sector, n, ref_of in (("IP", g.dims()[0], orc.ip_sigma), ("EA", g.dims()[1], orc.ea_sigma)):
        X = np.stack([random_vector(k + 1, n) + 1j * random_vector(k + 101, n) for k in range(nvec)])
        ref = np.stack([ref_of(x) for x in X])
        assert np.abs(g.sigma(sector, X) - ref).max() <= 1e-12 * np.abs(ref).max()
    g.close()


@pytest.mark.parametrize("flops", [0.0, 4e12, 1e18])
@pytest.mark.parametrize("o,v,L", [(1, 2, 3), (3, 7, 9), (7, 33, 41), (12, 61, 243)])
def test_setup_on_digit_planes(o, v, L, flops):
    """FP64 sigma of mixed-precision contexts whose set-up contractions (every order of strides the Hbar
    elements need) all run on digit planes, where they pay, or never: each within the FP64 bound."""
    pr = make_problem(o, v, L, seed=o + 5 * v, t1_std=0.05, t2_std=0.05, chol_sigma=0.3 if o < 10 else 0.05)
    gfcc.set_process_option(gfcc.OPT_SETUP_EMULATE_FLOPS, flops)
    try:
        g = gfcc.GFCC(pr, precision="mixed")
    finally:
        gfcc.set_process_option(gfcc.OPT_SETUP_EMULATE_FLOPS, 4e12)
    orc = GFCCOracle(pr.fock, pr.chol, pr.t1, pr.t2, o=o)
    for sector, n, ref_of in (("IP", g.dims()[0], orc.ip_sigma), ("EA", g.dims()[1], orc.ea_sigma)):
        x = random_vector(1, n) + 1j * random_vector(2, n)
        ref = ref_of(x)
        assert np.abs(g.sigma(sector, x)[0] - ref).max() <= 1e-12 * np.abs(ref).max()
    g.close()
