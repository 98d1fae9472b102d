"""The list radius of the Verlet-list build, in a wide box, pair by pair.

Pairs are planted at distances from 3.5e-6 to 3e-5 sigma inside and outside the
radius that the build tests (r_c + skin, widened by 1e-5 of it and 1e-6 of the
longest edge), apart along y and z, in a box of 1,000 sigma; the lists are read
from a checkpoint.  Each side's distance differs from the exact one by less
than 3e-6: 2 x 2.3e-7 from each position's fixed point (L / 2^32), ~5e-7 per
component from FP32 coordinates of at most two cell edges.  (Coordinates
counted from the box's corner would round by up to 3e-5 each.)
"""
import ctypes as C

import numpy as np
import pytest

from helpers import gpu, gpu_system

pytestmark = pytest.mark.gpu


def lists_of(P, path):
    """Ids and neighbour ids of every slot of a checkpoint without a reaction scheme."""
    raw = open(path, "rb").read()
    desc = P.prx_system_desc.from_buffer_copy(raw, 8)
    n, cap, at = desc.n, desc.adj_cap, 8 + C.sizeof(P.prx_system_desc)
    assert np.frombuffer(raw, np.int32, 1, at)[0] == 0  # no scheme
    at += 4 + C.sizeof(P.prx_reaction_desc) + 8
    nb = int(np.frombuffer(raw, np.uint64, 1, at)[0])
    at += 16
    ids = np.frombuffer(raw, np.uint32, n, at)
    at += 8 * n + 48 * n + 3 * n + 4 * n * cap + C.sizeof(P.prx_bond) * nb
    lcap = int(np.frombuffer(raw, np.int32, 1, at)[0])
    at += 4 + 4 * n
    nn = np.frombuffer(raw, np.uint8, n, at)
    at += n
    nl = np.frombuffer(raw, np.int32, lcap * n, at).reshape(lcap, n)
    assert at + 4 * lcap * n == len(raw)
    return ids, nn, nl


@pytest.mark.parametrize("shape", [(5.0, 1000.0, 1000.0), (1000.0, 1000.0, 5.0)])
def test_pairs_at_the_radius(tmp_path, shape):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    P = gpu()
    rng = np.random.default_rng(11)
    rv = 2.0 ** (1.0 / 6.0) + 0.3
    r = float(np.sqrt(float(np.float32((rv * (1 + 1e-5) + 1e-6 * max(shape)) ** 2))))
    wide = [d for d in range(3) if shape[d] > 100.0]
    m = 100  # sites along each long edge, 10 sigma apart: no two pairs meet
    site = np.stack(np.meshgrid(np.arange(m), np.arange(m), indexing="ij"), -1).reshape(-1, 2)
    a = np.full((m * m, 3), 2.5)
    a[:, wide] = (site + 0.5 + rng.uniform(-0.3, 0.3, site.shape)) * 10.0
    off = rng.choice([-1.0, 1.0], m * m) * rng.uniform(3.5e-6, 3e-5, m * m)
    t = rng.uniform(0.0, 2.0 * np.pi, m * m)
    d = np.zeros((m * m, 3))
    if 0 in wide:  # along the long edge that the build tests from its row's edges
        d[:, 1] = np.sign(np.cos(t))
    else:
        d[:, 1], d[:, 2] = np.cos(t), np.sin(t)
    b = (a + d * (r + off)[:, None]) % np.array(shape)
    x = np.concatenate([a, b])
    dx = b - a
    dx -= np.array(shape) * np.round(dx / np.array(shape))
    dist = np.sqrt((dx ** 2).sum(1))
    n = len(x)
    with gpu_system(P, shape, x, None, np.zeros(n, np.uint8), np.zeros(n, np.int8), cap=1, eps=0.0) as g:
        g.save(str(tmp_path / "c"))
    ids, nn, nl = lists_of(P, str(tmp_path / "c"))
    listed = np.zeros(n, bool)
    for k in range(int(nn.max())):
        has = nn > k
        partner = ids[nl[k][has]]
        assert np.all(np.abs(partner.astype(int) - ids[has].astype(int)) == m * m)
        listed[ids[has]] = True
    assert np.array_equal(listed[: m * m], listed[m * m:])
    # (cells have edges of r_c + skin or more: a pair at the widened radius can
    # lie two cells apart, where the build does not look)
    nc = np.floor(np.array(shape) / (rv * (1 + 1e-9)))
    apart = np.abs(np.floor(a / np.array(shape) * nc) - np.floor(b / np.array(shape) * nc))
    near = np.all((apart <= 1) | (apart == nc - 1), axis=1)
    wrong = listed[: m * m] != ((dist < r) & near)
    assert int(wrong.sum()) == 0, (np.flatnonzero(wrong)[:5], (dist - r)[wrong][:5], a[wrong][:5], b[wrong][:5])
