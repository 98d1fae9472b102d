"""prx_react_noalloc against prx_react_once at the edges of its ranges.

The allocation-free step shares its particles out over 128 blocks and the
warps of a block over its particles; the sizes sit at the edges of both.
Integer and FP64-decision work: tolerance zero.
"""
import numpy as np
import pytest

import synth
from helpers import canonical, gpu, gpu_reaction, gpu_system

pytestmark = pytest.mark.gpu
CAP = 4


@pytest.fixture(scope="module")
def torch():
    t = pytest.importorskip("torch")
    if not t.cuda.is_available():
        pytest.skip("no CUDA device")
    return t


def call(torch, P, rx, L, inp, x):
    n = inp.n
    dev = torch.device("cuda")
    pos, typ = torch.tensor(x, device=dev), torch.tensor(inp.type, device=dev)
    st = torch.tensor(inp.state, device=dev)
    nadj, adj = torch.zeros(n, dtype=torch.uint8, device=dev), torch.zeros(n * CAP, dtype=torch.int32, device=dev)
    out = torch.zeros(n * P.BOND_DTYPE.itemsize, dtype=torch.uint8, device=dev)
    nb = torch.zeros(1, dtype=torch.int32, device=dev)
    tr = P.prx_react_noalloc(rx, L, 0.005, 11, 10, n, pos.data_ptr(), typ.data_ptr(), st.data_ptr(), CAP,
                             nadj.data_ptr(), adj.data_ptr(), out.data_ptr(), n, nb.data_ptr(),
                             torch.cuda.current_stream().cuda_stream)
    return tr, canonical(out.cpu().numpy().view(P.BOND_DTYPE)[: int(nb.item())]), st.cpu().numpy()


@pytest.mark.parametrize("selection", [0, 1], ids=["random", "nearest"])
@pytest.mark.parametrize("n,share", [(2, 0.5), (127, 0.1), (129, 0.9), (1025, 0.01), (4097, 0.3), (16384, 0.1)])
def test_sizes(torch, n, share, selection):
    P = gpu()
    L = max(4.4, synth.box_edge(n))
    n_A = max(1, int(share * n))
    inp = synth.step_growth(n - n_A, n_A, 4, n, rho=n / L ** 3, jitter=0.5)
    rx = gpu_reaction(P, synth.step_growth_scheme(4, k=5.0, selection=selection))
    with gpu_system(P, L, inp.x, inp.v, inp.type, inp.state, cap=CAP, seed=11) as g:
        g.set_reaction(rx)
        ref = g.react_once(10), canonical(g.bonds()), g.states()
    assert n < 1000 or len(ref[1]) > 0  # the case is not vacuous
    # as they are, and all moved by whole box edges (outside the box the FP32 search is not used)
    for x in (inp.x, inp.x + 4.0 * L):
        got = call(torch, P, rx, L, inp, x)
        assert got[0] == ref[0]
        assert np.array_equal(got[1], ref[1]) and np.array_equal(got[2], ref[2])
