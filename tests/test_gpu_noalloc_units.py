"""prx_react_noalloc in units of length that leave the FP32 range when squared:
all lengths scaled by a power of two give the same decisions bit for bit (every
FP64 operation of the distance test scales exactly)."""
import numpy as np
import pytest

import synth
from helpers import gpu, gpu_reaction
from test_gpu_noalloc_sizes import call, torch  # noqa: F401 (torch is a fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("selection", [0, 1], ids=["random", "nearest"])
def test_scaled_lengths(torch, selection):  # noqa: F811
    P = gpu()
    inp = synth.step_growth(900, 100, 4, 3, jitter=0.5)
    L = float(inp.L)
    ref = call(torch, P, gpu_reaction(P, synth.step_growth_scheme(4, 5.0, selection=selection)), L, inp, inp.x)
    assert ref[0]["formed"] > 10
    for s in (-400, -130, -80, -62, -58, -20, 20, 55, 58, 62, 64, 80, 130, 400):
        rx = gpu_reaction(P, synth.step_growth_scheme(4, 5.0, selection=selection, r_react=float(np.ldexp(1.1, s))))
        got = call(torch, P, rx, float(np.ldexp(L, s)), inp, np.ldexp(inp.x, s))
        assert got[0] == ref[0], s
        assert np.array_equal(got[1], ref[1]) and np.array_equal(got[2], ref[2]), s
