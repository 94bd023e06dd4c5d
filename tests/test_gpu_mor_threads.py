"""Reduced models of different size used from two threads, each on a context of its own."""
import threading

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


def test_models_of_two_sizes_in_two_threads():
    # m about 60 and 96 with 6 right-hand sides: 64 and 158 KB of shared memory a block.  The larger one's calls launch
    # three times with a wait between, the smaller one's are short and many.
    orbs = np.arange(6)
    work = []
    for seed, samples, points, reps in ((1, 5, 2, 4000), (2, 8, 700, 60)):
        g = gfcc.GFCC(make_problem(6, 30, 60, seed=seed), sectors="IP", precision="mixed")
        mor = gfcc.MOR(g, "IP")
        mor.expand(np.linspace(-0.95, -0.25, samples), 0.05, orbs, 1e-8)
        assert 12 * samples - 4 < mor.dim() <= 12 * samples
        om = np.linspace(-1.0, -0.2, points)
        work.append((g, mor, om, reps, mor.green(om, 0.05, orbs, residuals=True)))
    bad = []

    def run(mor, om, reps, ref):
        for _ in range(reps):
            try:
                got = mor.green(om, 0.05, orbs, residuals=True)
                if not all(np.array_equal(a, b) for a, b in zip(got, ref)):
                    bad.append("differs")
            except gfcc.GFCCError as e:
                bad.append(str(e))

    th = [threading.Thread(target=run, args=w[1:]) for w in work]
    for t in th:
        t.start()
    for t in th:
        t.join()
    assert not bad, bad[:3]
    for g, mor, *_ in work:
        mor.close()
        g.close()
