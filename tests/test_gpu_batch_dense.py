"""Rebuilds of a batch whose members have many cells with more members than a
bucket holds: lookups go through the links of a cell's further members.  Bit for
bit as the members' runs alone, whose sort has no buckets (the member of 120,000
runs through the launch chain, the other through the persistent kernel)."""
import numpy as np
import pytest

import synth
from helpers import gpu, gpu_reaction, gpu_system

pytestmark = pytest.mark.gpu


def gas(P, n, per_cell, seed):
    """Particles without a pair force, `per_cell` per list-build cell on
    average, with 60 clumps of 17 to 24 inside a cell, apart; they react and bond."""
    rng = np.random.default_rng(seed)
    m = int(np.ceil((n / per_cell) ** (1.0 / 3.0)))
    L = m * (2.0 ** (1.0 / 6.0) + 0.3) * 1.0001
    x = rng.random((n, 3)) * L
    size = rng.integers(17, 25, 60)
    at = rng.choice((m // 3) ** 3, 60, replace=False)
    corner = 3 * np.stack([at % (m // 3), at // (m // 3) % (m // 3), at // (m // 3) ** 2], 1) * (L / m) + 0.4
    x[: size.sum()] = np.repeat(corner, size, axis=0) + 0.5 * rng.random((size.sum(), 3))
    typ = (np.arange(n) % 9 == 0).astype(np.uint8)
    g = gpu_system(P, L, x, rng.standard_normal((n, 3)), typ, np.where(typ == 1, 4, 0).astype(np.int8), cap=4,
                   seed=seed, eps=0.0)
    g.set_reaction(gpu_reaction(P, synth.step_growth_scheme(4, 0.3)))
    k = np.minimum((x / L * m).astype(int), m - 1)
    crowd = np.bincount((k[:, 2] * m + k[:, 1]) * m + k[:, 0], minlength=m ** 3)
    assert g.stats()["cells"] == (m, m, m) and (crowd > 16).sum() >= 60 and crowd.max() >= 24
    return g


def test_crowded_cells():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    P = gpu()
    specs = [(120000, 4.9, 1), (30000, 5.5, 2)]
    alone, members = [gas(P, *s) for s in specs], [gas(P, *s) for s in specs]
    with P.Batch() as b:
        for g in members:
            b.add(g)
        b.run(43)
        b.sync()
    for g, h in zip(alone, members):
        g.run(43)
        assert np.array_equal(g.positions(), h.positions()) and np.array_equal(g.velocities(), h.velocities())
        assert np.array_equal(g.states(), h.states()) and np.array_equal(g.bonds(), h.bonds())
        assert g.stats()["rebins"] == h.stats()["rebins"] > 3 and len(g.bonds()) > 1000
        g.close()
        h.close()
