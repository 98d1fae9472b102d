"""Device-driven runs (larger systems) against the one-phase kernels.

The step graph holds up to four steps, fewer for short reaction intervals and
for runs of fewer steps; what follows a step (a rebuild, a reaction step, the
run's end) may fall on any of them.  While profiling is on, prx_run launches
one kernel per phase from the host; both must give the same bits (tolerance
zero).
"""
import numpy as np
import pytest

import synth
from helpers import canonical, gpu, gpu_reaction, gpu_system

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return gpu()


@pytest.mark.parametrize("n,fp64,theta", [(80000, False, 0), (80000, False, 1), (80000, False, 2), (80000, False, 5),
                                          (80000, False, 10), (80000, False, 2 ** 32 - 1), (17000, True, 3),
                                          (17000, True, 9)])
def test_same_bits(P, n, fp64, theta):
    inp = synth.step_growth(n - n // 9, n // 9, 4, n)
    runs = (1, 2, 3, 4, 5, 9, 23)
    out = []
    for hosted in (False, True):
        with gpu_system(P, inp.L, inp.x, inp.v, inp.type, inp.state, cap=4, seed=n, fp64=fp64) as g:
            if theta:
                g.set_reaction(gpu_reaction(P, synth.step_growth_scheme(4, 10.0 / min(theta, 10), theta=theta)))
            if hosted:
                P.prx_profile_begin(g.h)
            for c in runs:
                g.run(c)
            if hosted:
                P.prx_profile_end(g.h)
            st = g.stats()
            out.append(dict(x=g.positions(), v=g.velocities(), bonds=canonical(g.bonds()), states=g.states(),
                            steps=st["steps"], reactions=st["reactions"], rebins=st["rebins"]))
    assert out[0]["steps"] == sum(runs) and out[0]["rebins"] > 2
    assert (len(out[0]["bonds"]) > 0) == (0 < theta <= sum(runs))
    for key in out[1]:
        assert np.array_equal(out[0][key], out[1][key]), key
