"""Which runs go through the persistent kernel: the cases whose results other
tests compare with the one-phase kernels' do, at both edges of the range, and
those beyond it do not.  The FP32 edge is one slot per thread of the GPU (512 per
SM), in FP64 mode 16,384."""
import ctypes as C

import numpy as np
import pytest

import synth
from helpers import gpu, gpu_reaction, gpu_system
from test_gpu_persistent import step_growth

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


def slots():
    import torch
    return 512 * torch.cuda.get_device_properties(0).multi_processor_count


@pytest.mark.parametrize("n,fp64,kw", [(1, False, {}), (31, False, {}), (4865, False, {}), (40000, False, {}),
                                       (1, True, {}), (609, True, {}), (1250, True, {}), (16384, True, {}),
                                       (700, False, {}), (3000, False, dict(selection=1, style=1))])
def test_in_range(P, n, fp64, kw):
    with step_growth(P, n, fp64=fp64, **kw)() as g:
        for c in (7, 33, 1):
            g.run(c)
        assert persistent_steps(P, g) == 41 == g.step()


@pytest.mark.parametrize("over", [0, 1])
def test_edges(P, over):
    for n, fp64 in ((slots() + over, False), (16384 + over, True)):
        with step_growth(P, n, fp64=fp64)() as g:
            g.run(12)
            assert persistent_steps(P, g) == (0 if over else 12) and g.step() == 12


def test_scheme_box_and_crowded_cells(P):
    inp = synth.step_growth_mixed(1500, 200, 100, 9)
    with gpu_system(P, inp.L, inp.x, inp.v, inp.type, inp.state, cap=6, seed=9) as g:
        g.set_reactions([gpu_reaction(P, s) for s in synth.concurrent_schemes(1.0, 3.0, 0.5)])
        g.run(20)
        assert persistent_steps(P, g) == 20
    inp, dims, cb = synth.ep_chains(300, 3, 4, 5)
    bonds = np.zeros(len(cb), P.BOND_DTYPE)
    bonds["a"], bonds["t"] = cb[:, 0], cb[:, 1]
    with gpu_system(P, dims, inp.x, inp.v, inp.type, inp.state, cap=4, seed=5, bonds=bonds) as g:
        g.run(20)
        assert persistent_steps(P, g) == 20
    rng = np.random.default_rng(4)
    n, L = 30000, 26.0
    x = rng.random((n, 3)) * L
    x[:24] = 5.2 + 0.5 * rng.random((24, 3))
    with gpu_system(P, L, x, None, np.zeros(n, np.uint8), np.zeros(n, np.int8), cap=4, seed=3, eps=0.0) as g:
        g.run(20)
        assert persistent_steps(P, g) == 20


def test_not_with_a_force_cap_four_lanes_or_profiling(P):
    inp = synth.step_growth(2700, 300, 4, 1)

    def make(**kw):
        return gpu_system(P, inp.L, inp.x, inp.v, inp.type, inp.state, cap=4, seed=1, **kw)
    with make(force_cap=100.0) as g, make() as h, make() as p:
        h.set_launch_config(step_lanes=4)
        P.prx_profile_begin(p.h)
        for s in (g, h, p):
            s.run(8)
        P.prx_profile_end(p.h)
        assert [persistent_steps(P, s) for s in (g, h, p)] == [0, 0, 0]
        h.set_launch_config()
        h.run(8)
        p.run(8)
        assert [persistent_steps(P, s) for s in (h, p)] == [8, 8]
