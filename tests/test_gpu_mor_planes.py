"""Model residuals of mixed-precision contexts (digit-plane products) against the same residuals in NumPy from
the model's own basis S, its image W = Hbar S and its model operator."""
import numpy as np
import pytest

from oracle import gfcc_ref as R
from paper_2010_04768_gb300 import gfcc
from paper_2010_04768_gb300.synthetic import make_problem

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="session", autouse=True)
def _built():
    from paper_2010_04768_gb300 import build
    build.build()
    gfcc.load()


# (1, 2): too small for the planes; 305 frequencies: a second launch of one frequency; 70 orbital-frequency pairs
# and n off the multiples of 64
@pytest.mark.parametrize("sector,n_om,n_orb", [("IP", 1, 2), ("IP", 305, 3), ("EA", 70, 7)])
def test_model_residuals_match_numpy(sector, n_om, n_orb):
    o, v, L, eta = 9, 37, 60, 0.02
    pr = make_problem(o, v, L, seed=3)
    orbs = np.arange(o - 4, o - 4 + n_orb, dtype=np.int32)
    samp = np.array([-0.9, -0.3]) if sector == "IP" else np.array([0.15, 0.6])
    g = gfcc.GFCC(pr, sectors=sector, precision="mixed")
    mor = gfcc.MOR(g, sector)
    _, code = mor.expand(samp, eta, orbs, 1e-9)
    assert code == gfcc.OK
    om = np.linspace(samp[0], samp[1], n_om) + 0.05
    _, rr = mor.green(om, eta, orbs, residuals=True)
    m = mor.dim()
    H, S = mor.projected(rows=m)
    W = g.sigma(sector, S)
    mor.close()
    g.close()
    sg = 1.0 if sector == "IP" else -1.0
    rhs = [R.ip_pack(*R.ip_rhs_unpacked(o, v, pr.t1, pr.t2, p)) if sector == "IP" else
           R.ea_pack(*R.ea_rhs_unpacked(o, v, pr.t1, pr.t2, p)) for p in orbs]
    B = np.stack(rhs)
    for w in {0, n_om // 2, n_om - 1}:
        z = om[w] + (-1j if sector == "IP" else 1j) * eta
        A = z * np.eye(m) + sg * H
        X = np.linalg.solve(A, (S @ B.T).astype(complex)).T
        r = B - (z * X) @ S - sg * X @ W
        ref = np.linalg.norm(r, axis=1) / np.linalg.norm(B, axis=1)
        # both sides round their solve: relative error cond(A) 2^-53 in X times ||A S X|| / ||b||, and m terms a sum
        size = (np.abs(z) * np.linalg.norm(X, axis=1) + np.linalg.norm(X @ W, axis=1)) / np.linalg.norm(B, axis=1)
        tol = 2.0 ** -53 * 4 * m * np.linalg.cond(A) * size
        assert np.all(np.abs(rr[w] - ref) <= tol)
