"""Persistent runs (prx_run of a small system) against the one-phase kernels.

While profiling is on, prx_run launches one kernel per phase; the persistent
kernel must give the same bits: positions, velocities, bonds, states, reaction
records and rebuild count (tolerance zero).  Sizes sit at the edges of its
chunks of 32 slots (4 in FP64 mode), its blocks and its range.
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


def result(g):
    st = g.stats()
    return dict(x=g.positions(), v=g.velocities(), bonds=canonical(g.bonds()), states=g.states(), hist=g.history(),
                reactions=np.array(st["reactions"]), rebins=np.array(st["rebins"]))


def assert_same_runs(P, make, chunks):
    """Runs the system made by `make` for each number of steps both ways."""
    with make() as g:
        for c in chunks:
            g.run(c)
        got = result(g)
    with make() as g:
        P.prx_profile_begin(g.h)
        for c in chunks:
            g.run(c)
        P.prx_profile_end(g.h)
        ref = result(g)
    for key in ref:
        assert np.array_equal(got[key], ref[key]), key
    return got


def step_growth(P, n, k=1.0, selection=0, fp64=False, f=4, style=0):
    L = max(4.4, synth.box_edge(n))
    inp = synth.step_growth(n - max(1, n // 9), max(1, n // 9), f, n, rho=n / L ** 3)

    def make():
        g = gpu_system(P, L, inp.x, inp.v, inp.type, inp.state, cap=f, seed=n, fp64=fp64)
        g.set_reaction(gpu_reaction(P, synth.step_growth_scheme(f, k, selection=selection, bond_style=style)))
        return g
    return make


@pytest.mark.parametrize("n", [1, 31, 33, 513, 4863, 4865, 40000, 77824, 77825])
def test_sizes(P, n):
    got = assert_same_runs(P, step_growth(P, n, f=6), (7, 33, 1))
    assert n < 500 or (len(got["bonds"]) > 0 and got["rebins"] > 3)


@pytest.mark.parametrize("n", [1, 3, 5, 607, 609, 1250])
def test_sizes_fp64(P, n):
    got = assert_same_runs(P, step_growth(P, n, fp64=True), (7, 34))
    assert n < 500 or (len(got["bonds"]) > 0 and got["rebins"] > 3)


@pytest.mark.parametrize("fp64", [False, True])
def test_more_steps_than_one_launch(P, fp64):
    """A run of several launches, and a reaction step at a launch's end."""
    assert_same_runs(P, step_growth(P, 700, fp64=fp64), (530,))


def test_nearest_rule_and_mirror_bonds(P):
    got = assert_same_runs(P, step_growth(P, 3000, selection=1, style=1), (60,))
    assert len(got["bonds"]) > 10


def test_concurrent_reactions(P):
    inp = synth.step_growth_mixed(1500, 200, 100, 9)

    def make():
        g = gpu_system(P, inp.L, inp.x, inp.v, inp.type, inp.state, cap=6, seed=9)
        g.set_reactions([gpu_reaction(P, s) for s in synth.concurrent_schemes(1.0, 3.0, 0.5)])
        return g
    assert len(assert_same_runs(P, make, (60,))["bonds"]) > 50


def test_box_that_is_not_cubic_with_chain_bonds(P):
    inp, dims, cb = synth.ep_chains(300, 3, 4, 5)
    bonds = np.zeros(len(cb), P.BOND_DTYPE)
    bonds["a"], bonds["t"] = cb[:, 0], cb[:, 1]

    def make():
        g = gpu_system(P, dims, inp.x, inp.v, inp.type, inp.state, cap=4, seed=5, bonds=bonds)
        g.set_reaction(gpu_reaction(P, synth.ep_scheme(4, 2.0)))
        return g
    assert_same_runs(P, make, (60,))


def test_crowded_cells(P):
    """Particles without a pair force, unevenly placed: cells with more
    members than a bucket holds and neighbour windows longer than a mask, which
    take the slower paths, beside ordinary ones; bonds form and pull."""
    rng = np.random.default_rng(4)
    n, L = 30000, 26.0
    x = rng.random((n, 3)) * L
    x[:24] = 5.2 + 0.5 * rng.random((24, 3))  # more than 24 in one cell
    typ = (np.arange(n) % 9 == 0).astype(np.uint8)
    st = np.where(typ == 1, 4, 0).astype(np.int8)

    def make():
        g = gpu_system(P, L, x, None, typ, st, cap=4, seed=3, eps=0.0)
        g.set_reaction(gpu_reaction(P, synth.step_growth_scheme(4, 0.5)))
        return g
    got = assert_same_runs(P, make, (60,))
    assert len(got["bonds"]) > 1000 and got["rebins"] > 3
