"""A closed-shell context holds no workspace of its digit-plane products between calls."""
import numpy as np
import pytest

from paper_2010_04768_gb300 import gfcc
from paper_2010_04768_gb300.synthetic import make_closed_shell_problem, random_vector

pytestmark = pytest.mark.gpu


def test_workspace_is_given_back():
    torch = pytest.importorskip("torch")
    from paper_2010_04768_gb300 import build
    build.build()
    pr, orbs = make_closed_shell_problem(16, 80, 60, seed=5), np.arange(8, 16)

    def calls(g):
        x = np.stack([random_vector(k, g.dims()[0]) + 1j * random_vector(50 + k, g.dims()[0]) for k in range(8)])
        g.sigma("IP", x)
        g.solve([-0.6], 0.01, orbs, 1e-6)
        torch.cuda.synchronize()
        return torch.cuda.mem_get_info()[0]

    warm = gfcc.GFCC(pr, sectors="IP", closed_shell=True)   # loads the kernels
    calls(warm)
    warm.close()
    g = gfcc.GFCC(pr, sectors="IP", closed_shell=True)
    g.set_option(gfcc.OPT_CLOSED_SHELL_EMULATE, 0)
    free = calls(g)                                          # what the context keeps without digit planes
    g.set_option(gfcc.OPT_CLOSED_SHELL_EMULATE, 1)
    assert calls(g) == free
    g.close()
