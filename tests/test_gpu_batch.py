"""gfcc_solve_batch on mixed-precision contexts: molecules of o = 10 to 19 solved together, over and over and with new
contexts between, give what each gives alone."""
import numpy as np
import pytest

from paper_2010_04768_gb300 import gfcc
from paper_2010_04768_gb300.synthetic import make_problem

pytestmark = pytest.mark.gpu


def test_uneven_mixed_molecules_together():
    from paper_2010_04768_gb300 import build
    build.build()
    om, eta, tol = np.linspace(-0.95, -0.35, 4), 0.005, 1e-8
    sets = []
    for seed in range(3):
        ctxs = [gfcc.GFCC(make_problem(o, 5 * o, 8 * o, seed=seed), sectors="IP", precision="mixed")
                for o in (10, 13, 16, 19)]
        sets.append((ctxs, [(om, eta, np.arange(c.o - 8, c.o), tol) for c in ctxs]))
    first = [gfcc.solve_batch(*s) for s in sets]       # shapes that no solve alone has met
    alone = [[c.solve(*r) for c, r in zip(*s)] for s in sets]
    for rep in range(40):
        for k, s in enumerate(sets):
            Gs, codes = first[k] if rep == 0 else gfcc.solve_batch(*s)
            for G, code, (ref, ref_code) in zip(Gs, codes, alone[k]):
                assert code == ref_code == gfcc.OK
                # either is within tol |b| |c| / eta of the exact values (|A^-1| <= 1 / eta), |b| |c| about 1.2
                assert np.abs(G - ref).max() <= 2.5 * tol / eta
    for ctxs, _ in sets:
        for c in ctxs:
            c.close()
