"""A persistent run whose barrier gives up: PRX_ETIMEOUT is reported, and what
the interrupted rebuild left (cell counters that are not zero, positions in the
next set's order) is never built upon: runs queued behind it do nothing, later
ones are refused, and a batch that the system was queued into before anyone knew
keeps its other members' results.

The barrier is made to give up by a limit of one poll on ordinary runs.
"""
import ctypes as C

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


def make(P, n, fp64=False, polls=0):
    inp = synth.step_growth(n - n // 9, n // 9, 4, n)
    g = gpu_system(P, inp.L, inp.x, inp.v, inp.type, inp.state, cap=4, seed=n, fp64=fp64)
    g.set_reaction(gpu_reaction(P, synth.step_growth_scheme(4, 1.0)))
    if polls:
        assert P.lib().prx_test_wait_limit(g.h, C.c_uint32(polls)) == P.PRX_OK
    return g


def step_of(P, g):
    s = C.c_uint64()
    rc = P.lib().prx_get_step(g.h, C.byref(s))
    return rc, s.value


@pytest.mark.parametrize("n,fp64", [(4863, False), (33000, False), (1250, True)])
def test_status_and_later_runs(P, n, fp64):
    with make(P, n, fp64, polls=1) as g:
        for _ in range(3):  # the first launch gives up; the others are queued behind it
            g.run(100)
        rc, step = step_of(P, g)
        assert rc == P.PRX_ETIMEOUT and 1 <= step <= 100
        for call in (lambda: g.run(1), g.sync, lambda: g.run(0)):
            with pytest.raises(P.PolyrxError) as e:
                call()
            assert e.value.code == P.PRX_ETIMEOUT
        with P.Batch() as b, pytest.raises(P.PolyrxError) as e:
            b.add(g)
        assert e.value.code == (P.PRX_EINVAL if fp64 else P.PRX_ETIMEOUT)  # (batches take no FP64 system)
        assert step_of(P, g) == (P.PRX_ETIMEOUT, step)
        # read-backs still return every particle once (a garbled state, in its place)
        x = np.zeros((n, 3))
        assert P.lib().prx_get_positions(g.h, x.ctypes.data_as(C.c_void_p)) == P.PRX_ETIMEOUT


def test_other_routes_do_not_rebuild(P):
    """The launch chain and a batch queued behind the run, before its status is known."""
    with make(P, 4863, polls=1) as g, make(P, 3000) as h, make(P, 3000) as ref:
        g.run(100)
        g.set_launch_config(step_threads=128, step_lanes=4)  # the chain's kernels
        P.lib().prx_run(g.h, C.c_uint64(40))  # (taken or refused: the status may not be known yet)
        assert step_of(P, g)[0] == P.PRX_ETIMEOUT
        with make(P, 4863, polls=1) as q, P.Batch() as b:
            q.run(100)
            assert b.admit(q, 40) is not None and b.admit(h, 40) is not None
            while b.step_epoch(40):
                pass
            assert P.lib().prx_sync(q.h) == P.PRX_ETIMEOUT
            h.sync()
            ref.run(40)
            assert np.array_equal(h.positions(), ref.positions()) and np.array_equal(h.bonds(), ref.bonds())
            b.poll()


def test_an_ordinary_limit_changes_nothing(P):
    with make(P, 4863) as g, make(P, 4863, polls=1 << 22) as h:
        g.run(60)
        h.run(60)
        assert np.array_equal(g.positions(), h.positions()) and np.array_equal(g.bonds(), h.bonds())
        assert P.lib().prx_test_wait_limit(g.h, C.c_uint32(0)) == P.PRX_EINVAL
