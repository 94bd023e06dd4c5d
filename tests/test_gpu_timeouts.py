"""Calls whose tensor-core products cannot finish report GFCC_ERR_TIMEOUT, and soon.

As in test_gpu_failure.py the bounded waits are made to run out on the host's order: their producers issue no loads
(GFCC_OPT_TEST_NO_LOADS) and the limit (GFCC_OPT_WAIT_NS) is short.  Afterwards the same calls give what they gave before.
"""
import time
from contextlib import contextmanager

import numpy as np
import pytest

from paper_2010_04768_gb300 import gfcc
from paper_2010_04768_gb300.synthetic import make_closed_shell_problem, make_problem, random_vector

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2010_04768_gb300 import build
    build.build()
    gfcc.load()


@contextmanager
def no_loads(wait_ns):
    gfcc.set_process_option(gfcc.OPT_AUTOTUNE, 0.0)   # no tile is chosen from launches that do nothing
    gfcc.set_process_option(gfcc.OPT_WAIT_NS, wait_ns)
    gfcc.set_process_option(gfcc.OPT_TEST_NO_LOADS, 1.0)
    try:
        yield
    finally:
        gfcc.set_process_option(gfcc.OPT_TEST_NO_LOADS, 0.0)
        gfcc.set_process_option(gfcc.OPT_WAIT_NS, 1e9)
        gfcc.set_process_option(gfcc.OPT_AUTOTUNE, 1.0)


def timed_out(call, wait_ns=2000.0, within=None):
    t = time.perf_counter()
    with no_loads(wait_ns):
        with pytest.raises(gfcc.GFCCError) as e:
            call()
    assert e.value.code == gfcc.ERR_TIMEOUT
    if within is not None:
        assert time.perf_counter() - t < within


@pytest.mark.parametrize("guess", [False, True])
def test_mixed_solve_ends_after_about_one_limit(guess):
    # 20 ms a wait: the products of one Arnoldi step alone would take 0.1 s one after the other, a refinement of 60
    # steps 6 s
    om, orbs = [-0.7, -0.6], [0, 3, 5]
    g = gfcc.GFCC(make_problem(6, 30, 60, seed=4), sectors="IP", precision="mixed")
    if guess:
        g.set_option(gfcc.OPT_GUESS, gfcc.GUESS_MINRES)
    other = gfcc.GFCC(make_problem(5, 24, 50, seed=5), sectors="IP", precision="mixed")
    ref, ref_other = g.solve(om, 0.01, orbs, 1e-9)[0], other.solve(om, 0.01, [1, 2], 1e-9)[0]
    timed_out(lambda: g.solve(om, 0.01, orbs, 1e-9), wait_ns=2e7, within=1.5)
    # neither another context nor this one's next call sees it
    for k, (a, b) in ((other, ([1, 2], ref_other)), (g, (orbs, ref))):
        G, code = k.solve(om, 0.01, a, 1e-9)
        assert code == gfcc.OK and np.abs(G - b).max() <= 1e-7 * np.abs(b).max()
    g.close()
    other.close()


def test_mixed_context_creation():
    pr = make_problem(6, 40, 80, seed=3)
    timed_out(lambda: gfcc.GFCC(pr, sectors="IP+EA", precision="mixed"))
    g = gfcc.GFCC(pr, sectors="IP", precision="mixed")
    assert g.solve([-0.5], 0.01, [0, 1, 2], 1e-9)[1] == gfcc.OK
    g.close()


def test_emulated_ccsd():
    pr = make_problem(6, 40, 60, seed=3)

    def call():
        return gfcc.ccsd(pr.fock, pr.chol, pr.o, tol=1e-8, want_lambda=True, emulate=True)

    ref = call()
    timed_out(call)
    got = call()
    assert got[-1] == ref[-1] and all(np.array_equal(a, b) for a, b in zip(got[:4], ref[:4]))


def test_closed_shell_operator():
    g = gfcc.GFCC(make_closed_shell_problem(10, 60, 100, seed=2), sectors="IP", closed_shell=True)
    x = np.stack([random_vector(k, g.dims()[0]) + 1j * random_vector(20 + k, g.dims()[0]) for k in range(8)])
    orbs = np.arange(2, 10)
    ref, G0 = g.sigma("IP", x), g.solve([-0.6], 0.01, orbs, 1e-8)[0]
    timed_out(lambda: g.sigma("IP", x))
    timed_out(lambda: g.solve([-0.6], 0.01, orbs, 1e-8))
    assert np.array_equal(g.sigma("IP", x), ref)
    assert np.array_equal(g.solve([-0.6], 0.01, orbs, 1e-8)[0], G0)
    g.close()


def test_tuning_keeps_no_choice_from_launches_that_gave_up():
    # a shape of its own whose first call times out: the next one times its tiles again, the one after that does not
    rng = np.random.default_rng(9)
    A, B = rng.standard_normal((391, 517), dtype=np.float32), rng.standard_normal((263, 517), dtype=np.float32)
    n = gfcc.launch_count()
    gfcc.set_process_option(gfcc.OPT_WAIT_NS, 2000.0)
    gfcc.set_process_option(gfcc.OPT_TEST_NO_LOADS, 1.0)
    try:
        with pytest.raises(gfcc.GFCCError) as e:
            gfcc.selftest_gemm_bf16(A, B)
    finally:
        gfcc.set_process_option(gfcc.OPT_TEST_NO_LOADS, 0.0)
        gfcc.set_process_option(gfcc.OPT_WAIT_NS, 1e9)
    assert e.value.code == gfcc.ERR_TIMEOUT
    tried = gfcc.launch_count() - n
    n = gfcc.launch_count()
    first = gfcc.selftest_gemm_bf16(A, B)
    assert gfcc.launch_count() - n >= tried > 2      # timed again: the tiles, then the product
    n = gfcc.launch_count()
    assert np.array_equal(gfcc.selftest_gemm_bf16(A, B), first) and gfcc.launch_count() - n == 1


def test_host_wait_gives_up():
    gfcc.selftest_host_wait(0.0)
    gfcc.selftest_host_wait(0.3)
    gfcc.set_process_option(gfcc.OPT_WAIT_NS, 2000.0)   # the host's limit: 2 s
    try:
        with pytest.raises(gfcc.GFCCError) as e:
            gfcc.selftest_host_wait(2.5)
    finally:
        gfcc.set_process_option(gfcc.OPT_WAIT_NS, 1e9)
    assert e.value.code == gfcc.ERR_TIMEOUT
    gfcc.selftest_host_wait(2.5)
