"""Small systems run at once, each on its own stream.  A few go through the
persistent kernel, one after the other; many through their launch chains, which
share the GPU, and back through the persistent kernel once they run alone.  The
results are those of each system alone, bit for bit."""
import ctypes as C
import threading
import time

import numpy as np
import pytest

from helpers import gpu
from test_gpu_persistent import result, step_growth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return gpu()


def persistent_steps(P, g):
    k = C.c_uint64()
    assert P.lib().prx_test_persistent_steps(g.h, C.byref(k)) == P.PRX_OK
    return k.value


def alone(make, runs):
    with make() as g:
        for c in runs:
            g.run(c)
            g.sync()
        return result(g)


def close(gs):
    for g in gs:
        g.close()


@pytest.mark.parametrize("n,k,fp64", [(2000, 8, False), (33000, 6, False), (9000, 6, True)])
def test_many_at_once(P, n, k, fp64):
    runs = (600, 300, 301)
    make = step_growth(P, n, fp64=fp64)
    ref = alone(make, runs)
    gs = [make() for _ in range(k)]
    for c in runs:
        for g in gs:
            g.run(c)
        for g in gs:
            g.sync()
    took = [persistent_steps(P, g) for g in gs]
    # the last one queued found the others under way, the first from its second run on
    assert took[0] == 600 and took[-1] == 0, took
    for g in gs:
        got = result(g)
        for key in ref:
            assert np.array_equal(got[key], ref[key]), key
    # alone again: one more run takes the chain, the next ones do not
    g = gs[0]
    for c in (5, 20, 7):
        g.run(c)
        g.sync()
    assert persistent_steps(P, g) == took[0] + 27
    close(gs)


def test_two_at_once(P):
    make = step_growth(P, 2000)
    gs = [make() for _ in range(2)]
    for _ in range(3):
        for g in gs:
            g.run(300)
        for g in gs:
            g.sync()
    assert [persistent_steps(P, g) for g in gs] == [900, 900]
    close(gs)


@pytest.mark.parametrize("n,took", [(2000, 400), (33000, 0)])
def test_beside_a_large_system(P, n, took):
    make = step_growth(P, n)
    ref = alone(make, (400,))
    with step_growth(P, 300000)() as big, make() as g:
        big.run(400)
        g.run(400)
        assert persistent_steps(P, g) == took
        got = result(g)
        for key in ref:
            assert np.array_equal(got[key], ref[key]), key
        big.sync()


def test_first_chains_return_without_waiting(P):
    """New systems whose chains are made while a persistent launch has the GPU: a
    launch of 512 steps takes about 19 ms here, a call that waits for its end up to
    as long; the limit is a quarter of that.  (The first round loads the kernels.)"""
    make = step_growth(P, 16000, fp64=True)
    for _ in range(2):
        gs = [make() for _ in range(8)]
        for g in gs:
            g.sync()
        calls = []
        for g in gs:
            t = time.perf_counter()
            g.run(2000)
            calls.append(time.perf_counter() - t)
        for g in gs:
            g.sync()
        assert persistent_steps(P, gs[0]) == 2000 and persistent_steps(P, gs[-1]) == 0
        close(gs)
    assert max(calls) < 5e-3, calls


def test_destroyed_while_others_run(P):
    """A system leaves with its run under way: it counts no longer."""
    make = step_growth(P, 2000)
    gs = [make() for _ in range(8)]
    for g in gs:
        g.run(200)
    close(gs)
    with make() as g:
        g.run(50)
        assert persistent_steps(P, g) == 50


def test_threads(P):
    """One thread per system, as a program that serves several users would."""
    make = step_growth(P, 1500)
    runs = (150, 40, 211)
    ref = alone(make, runs)
    got = [None] * 6

    def work(q):
        with make() as g:
            for c in runs:
                g.run(c)
            got[q] = result(g)

    ts = [threading.Thread(target=work, args=(q,)) for q in range(len(got))]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    for r in got:
        for key in ref:
            assert np.array_equal(r[key], ref[key]), key
