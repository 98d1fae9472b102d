"""prx_get_bonds returns the bond list in canonical order (step, a, t) at the
edges of the device sort: single records, one tile of 1,024, a run more, the
last run alone, equal records, steps that do not ascend and negative ones."""
import numpy as np
import pytest

from helpers import gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m", [1, 2, 1023, 1024, 1025, 2049, 5000])
def test_initial_bonds_come_back_sorted(m):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    P = gpu()
    rng = np.random.default_rng(m)
    n, L = 6000, 40.0
    x = rng.random((n, 3)) * L
    bonds = np.zeros(m, P.BOND_DTYPE)
    # each particle in at most two bonds: a ring, shuffled, so that the adjacency holds them
    ring = rng.permutation(n)
    at = rng.permutation(n)[:m]
    bonds["a"], bonds["t"] = ring[at], ring[(at + 1) % n]
    bonds["step"] = rng.integers(-3, 4, m) * 10
    bonds["style"] = rng.integers(0, 2, m)
    bonds["reaction"] = np.arange(m)  # tells equal keys apart
    if m > 4:  # equal (step, a, t) with other styles: they keep their order
        bonds[["a", "t", "step"]][:2] = bonds[["a", "t", "step"]][2:4]
        for f in ("a", "t", "step"):
            bonds[f][m - 1] = bonds[f][0]
    desc = P.make_desc(n, L, adj_cap=4)
    with P.System(desc, x, None, np.zeros(n, np.uint8), np.zeros(n, np.int8), bonds=bonds) as g:
        want = bonds[np.lexsort((bonds["reaction"], bonds["t"], bonds["a"], bonds["step"]))]
        assert np.array_equal(g.bonds(), want)
        assert np.array_equal(g.bonds(), want)  # the list itself is still whole
        short = np.zeros(m, P.BOND_DTYPE)[: max(1, m // 2)]
        import ctypes
        k = ctypes.c_uint64()
        rc = P.lib().prx_get_bonds(g.h, short.ctypes.data, len(short), ctypes.byref(k))
        assert k.value == m and rc == (P.PRX_ECAPACITY if len(short) < m else P.PRX_OK)
        assert np.array_equal(short, want[: len(short)])
