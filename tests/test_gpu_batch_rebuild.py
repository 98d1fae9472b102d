"""Rebuilds of a batch against the members' runs alone, bit for bit: cells with
more members than a bucket holds, and a member whose cells have no buckets
(which takes the whole batch through the ten-kernel rebuild)."""
import numpy as np
import pytest

import synth
from helpers import gpu, gpu_reaction, gpu_system

pytestmark = pytest.mark.gpu


def gas(P, n, L, seed, clump):
    """Particles without a pair force that react and bond."""
    rng = np.random.default_rng(seed)
    x = rng.random((n, 3)) * L
    if clump:
        x[:24] = 5.2 + 0.5 * rng.random((24, 3))
    typ = (np.arange(n) % 9 == 0).astype(np.uint8)
    g = gpu_system(P, L, x, None, typ, np.where(typ == 1, 4, 0).astype(np.int8), cap=4, seed=seed, eps=0.0)
    g.set_reaction(gpu_reaction(P, synth.step_growth_scheme(4, 0.3)))
    return g


@pytest.mark.parametrize("dense", [False, True], ids=["buckets", "no_buckets"])
def test_members_equal_their_runs_alone(dense):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    P = gpu()
    specs = [(3000, 17.0, 1, False), (30000, 26.0, 2, True), (257, 9.0, 3, False)]
    if dense:
        specs.append((9000, 14.0, 4, False))
    alone, members = [gas(P, *s) for s in specs], [gas(P, *s) for s in specs]
    with P.Batch() as b:
        for g in members:
            b.add(g)
        b.run(53)
        b.sync()
    for g, h in zip(alone, members):
        g.run(53)
        assert np.array_equal(g.positions(), h.positions()) and np.array_equal(g.velocities(), h.velocities())
        assert np.array_equal(g.states(), h.states()) and np.array_equal(g.bonds(), h.bonds())
        assert g.stats()["rebins"] == h.stats()["rebins"] > 3 and len(g.bonds()) > 0
        g.close()
        h.close()
