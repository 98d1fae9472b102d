"""Persistent runs of several launches, which the device drives: the same bits as
the same steps in runs of one launch each, in any mixture of the two and across a
change of the reaction scheme; and prx_run returns without waiting, however much
is queued."""
import time

import numpy as np
import pytest

import synth
from helpers import gpu, gpu_reaction, gpu_system

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return gpu()


def make(P, n, fp64=False):
    L = max(4.4, synth.box_edge(n))
    inp = synth.step_growth(n - max(1, n // 9), max(1, n // 9), 4, n, rho=n / L ** 3)
    return gpu_system(P, L, inp.x, inp.v, inp.type, inp.state, cap=4, seed=n, fp64=fp64)


@pytest.mark.parametrize("n,fp64", [(1, False), (2000, False), (30000, False), (1250, True)])
def test_same_bits(P, n, fp64):
    out = []
    for whole in (True, False):
        with make(P, n, fp64) as g:
            for scheme, runs in ((0.5, (513, 3, 512, 600, 1025)), (0.1, (511, 514, 1)), (None, (700,))):
                g.set_reaction(gpu_reaction(P, synth.step_growth_scheme(4, scheme)) if scheme else None)
                for c in runs:
                    while c > 100 and not whole:
                        g.run(100)
                        c -= 100
                    g.run(c)
            st = g.stats()
            out.append((g.positions(), g.velocities(), g.bonds(), g.states(), g.history(), st["steps"], st["rebins"]))
    for a, b in zip(*out):
        assert np.array_equal(a, b)
    assert out[0][5] == 4379 and (n < 500 or len(out[0][2]) > 100)


def test_returns_without_waiting(P):
    with make(P, 64) as g:
        g.run(1000)
        g.sync()
        t = time.perf_counter()
        for _ in range(5):
            g.run(100000)
        queued = time.perf_counter() - t
        g.sync()
        total = time.perf_counter() - t
        assert g.step() == 501000
    assert queued < 0.2 * total, (queued, total)


def test_a_timeout_ends_the_run(P):
    import ctypes as C
    with make(P, 4863) as g:
        assert P.lib().prx_test_wait_limit(g.h, C.c_uint32(1)) == P.PRX_OK
        g.run(3000)
        step = C.c_uint64()
        assert P.lib().prx_get_step(g.h, C.byref(step)) == P.PRX_ETIMEOUT and 1 <= step.value <= 512
