"""The BF16 operator against the FP64 one at odd and even orbital counts and past the ends of its tiles (32 virtual
orbitals, 16 or 32 pairs of occupied ones), where the layouts of the unpacked vector change their alignment."""
import numpy as np
import pytest

from paper_2010_04768_gb300 import gfcc
from paper_2010_04768_gb300.synthetic import make_problem

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="session", autouse=True)
def _built():
    from paper_2010_04768_gb300 import build
    build.build()
    gfcc.load()


@pytest.mark.parametrize("o,v", [(2, 3), (3, 5), (4, 32), (5, 33), (7, 64), (30, 31), (31, 32), (32, 33), (35, 36), (3, 35)])
@pytest.mark.parametrize("sector", ["IP", "EA"])
@pytest.mark.parametrize("nvec", [1, 3])
def test_mixed_sigma_matches_fp64(o, v, sector, nvec):
    pr = make_problem(o, v, o + v, seed=1)
    g = gfcc.GFCC(pr, sectors=sector, precision="mixed")
    n = g.dims()[0 if sector == "IP" else 1]
    rng = np.random.default_rng(o * 100 + v)
    X = rng.standard_normal((nvec, n)) + 1j * rng.standard_normal((nvec, n))
    ref = g.sigma(sector, X)
    got = g.sigma(sector, X, precision="mixed")
    g.close()
    # both operands rounded to 8 bits (2^-9 each, relative to their own size): 4 x the rms of a sum of such products;
    # a misplaced column of a tile is an error of 1 / sqrt(32) and more
    assert np.linalg.norm(got - ref) <= 4 * 2.0 ** -8 * np.linalg.norm(ref)


@pytest.mark.parametrize("o,v", [(2, 3), (3, 5), (4, 32), (5, 33), (30, 31), (31, 32), (35, 36), (3, 35)])
@pytest.mark.parametrize("sector", ["IP", "EA"])
def test_refined_solution_matches_fp64(o, v, sector):
    # the digit planes of the residual: a wrong digit of a layout leaves a residual above the tolerance, which the
    # FP64 solution shows
    pr = make_problem(o, v, o + v, seed=2)
    om, eta, orbs = [-0.4 if sector == "IP" else 0.4], 0.2, np.arange(o - 1, o + 1, dtype=np.int32)
    G = {}
    for prec in ("fp64", "mixed"):
        g = gfcc.GFCC(pr, sectors=sector, precision=prec)
        G[prec], code = g.solve(om, eta, orbs, 1e-11)
        g.close()
        assert code == gfcc.OK
    # two solutions within 1e-11 of ||b|| in the residual, the resolvent bounded by 1 / eta times the conditioning of
    # the non-normal operator (10 covers it at these sizes)
    assert np.abs(G["mixed"] - G["fp64"]).max() <= 2 * 1e-11 / eta * 10 * max(1.0, np.abs(G["fp64"]).max())
