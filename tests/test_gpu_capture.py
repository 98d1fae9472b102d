"""prx_run on a stream that is being captured into a CUDA graph is refused, for
every route of a run; the capture and the system go on as if it had not been
called."""
import ctypes as C

import numpy as np
import pytest

import synth
from helpers import gpu, gpu_reaction

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,fp64", [(2048, False), (1250, True), (80000, False)])
def test_run_is_refused_while_capturing(n, fp64):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    P = gpu()
    inp = synth.step_growth(n - n // 9, n // 9, 4, n)
    stream = torch.cuda.Stream()
    y = torch.zeros(4, device="cuda")
    out = []
    for captured in (False, True):
        desc = P.make_desc(n, inp.L, adj_cap=4, seed=n, fp64=fp64)
        with P.System(desc, inp.x, inp.v, inp.type, inp.state, stream=stream.cuda_stream) as g:
            g.set_reaction(gpu_reaction(P, synth.step_growth_scheme(4, 1.0)))
            g.run(12)
            if captured:
                graph = torch.cuda.CUDAGraph()
                with torch.cuda.graph(graph, stream=stream, capture_error_mode="thread_local"):
                    assert P.lib().prx_run(g.h, C.c_uint64(10)) == P.PRX_ECUDA
                    assert b"captured" in P.lib().prx_last_error(g.h)
                    y += 1.0
                    assert P.lib().prx_run(g.h, C.c_uint64(300)) == P.PRX_ECUDA
                graph.replay()
                torch.cuda.synchronize()
                assert y.tolist() == [1.0] * 4
            for c in (1, 20, 7):
                g.run(c)
            out.append((g.positions(), g.bonds(), g.step(), g.stats()["rebins"]))
    for a, b in zip(*out):
        assert np.array_equal(a, b)
    assert out[0][2] == 40 and len(out[0][1]) > 0
