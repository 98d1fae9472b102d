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


HISTOGRAM = """
import ctypes as C, sys
sys.path.insert(0, "tests")
import numpy as np, torch
import synth
from helpers import gpu
P = gpu()
n = 2048
inp = synth.step_growth(n - 200, 200, 4, 1)
stream = torch.cuda.Stream()
g = P.System(P.make_desc(n, inp.L, adj_cap=4), inp.x, inp.v, inp.type, inp.state, stream=stream.cuda_stream)
a = P.prx_class(1, 0, 15)
def histogram(counts):
    k = C.c_uint64(99)
    rc = P.lib().prx_pair_histogram(g.h, C.byref(a), C.byref(a), 1.1, len(counts), counts.ctypes.data, C.byref(k), C.byref(k))
    return rc, k.value
c = np.zeros(50, np.uint64)
assert histogram(c) == (P.PRX_OK, n - 200) and c.sum() > 0
graph = torch.cuda.CUDAGraph()
c[:] = 7
with torch.cuda.stream(stream):
    graph.capture_begin(capture_error_mode="thread_local")
    rc, k = histogram(c)  # its wait is refused, which also ends the capture
assert rc == P.PRX_ECUDA and k == 99 and (c == 7).all(), (rc, k, c)
print("untouched", flush=True)
import os
os._exit(0)
"""


def test_a_failed_histogram_writes_nothing():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import os
    import subprocess
    import sys
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", HISTOGRAM], cwd=root, capture_output=True, text=True, timeout=240)
    assert r.returncode == 0 and "untouched" in r.stdout, r.stdout + r.stderr
