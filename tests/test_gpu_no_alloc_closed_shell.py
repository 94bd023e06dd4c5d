"""gfcc_sigma_noalloc on a closed-shell context takes no device memory, at sizes whose products gfcc_sigma evaluates from
digit planes (which need a workspace)."""
import numpy as np
import pytest

from paper_2010_04768_gb300 import gfcc
from paper_2010_04768_gb300.synthetic import make_closed_shell_problem, random_vector

pytestmark = pytest.mark.gpu


def test_closed_shell_sigma_noalloc_takes_no_memory():
    torch = pytest.importorskip("torch")
    from paper_2010_04768_gb300 import build
    build.build()
    o, v = 10, 80                  # contraction length o o v = 8000, just below the limit of the call
    g = gfcc.GFCC(make_closed_shell_problem(o, v, 40, seed=5), sectors="IP", closed_shell=True)
    n = g.dims()[0]
    X = np.stack([random_vector(k, n) + 1j * random_vector(50 + k, n) for k in range(3)])
    x_dev = torch.from_numpy(X.view(np.float64).copy()).cuda()
    y_dev = torch.full_like(x_dev, float("nan"))
    g.set_option(gfcc.OPT_CLOSED_SHELL_EMULATE, 0)
    ref = g.sigma("IP", X)
    g.sigma_noalloc("IP", X.shape[0], x_dev.data_ptr(), y_dev.data_ptr())   # loads its kernels
    g.set_option(gfcc.OPT_CLOSED_SHELL_EMULATE, 1)
    y_dev.fill_(float("nan"))
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    g.sigma_noalloc("IP", X.shape[0], x_dev.data_ptr(), y_dev.data_ptr())
    assert torch.cuda.mem_get_info()[0] == free
    Y = y_dev.cpu().numpy().view(np.complex128).reshape(X.shape)
    assert np.abs(Y - ref).max() <= 1e-12 * np.abs(ref).max()
    g.close()
