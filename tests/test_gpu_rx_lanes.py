"""Reaction steps over the numbers of eligible A's at which the search and the
selection change their lanes per A (16, 4, 1; 4, 1): bit for bit the oracle's
bonds and states for the nearest-partner rule, concurrent reactions and the
random rule, from a state with many competitors per T (p near 1).  (The concurrent search
has one lane beyond 200,000.)"""
import numpy as np
import pytest

import oracle as orc
import synth
from helpers import bonds_of_oracle, canonical, gpu, gpu_reaction, gpu_system, md_params, orc_reaction, oracle_system

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rule", ["random", "nearest", "concurrent"])
@pytest.mark.parametrize("n_a", [3, 4999, 5001, 19999, 20001, 32768, 32770, 90001, 200003])
def test_reaction_step(rule, n_a):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    P = gpu()
    n_b = max(600, n_a)
    if rule == "concurrent":
        inp = synth.step_growth_mixed(n_b, n_a - n_a // 3, n_a // 3, n_a, jitter=0.5)
        sch = synth.concurrent_schemes(18.0, 9.0, 14.0)
    else:
        inp = synth.step_growth(n_b, n_a, 4, n_a, jitter=0.5)
        sch = [synth.step_growth_scheme(4, 18.0, selection=int(rule == "nearest"))]
    eligible = int(((inp.type != 0) & (inp.state > 0)).sum())
    assert eligible == n_a
    o = oracle_system(inp.x, inp.v, inp.type, inp.state, 6)
    md = md_params(inp.L, 7)
    with gpu_system(P, inp.L, inp.x, inp.v, inp.type, inp.state, cap=6, seed=7) as g:
        g.set_reactions([gpu_reaction(P, s) for s in sch])
        for step in (10, 20):
            tr = g.react_once(step)
            if len(sch) > 1:
                ref, _ = orc.react_set(o, md, [orc_reaction(s) for s in sch], step, use_cells=True)
            else:
                ref = orc.react(o, md, orc_reaction(sch[0]), step, use_cells=True)
            assert tr == ref
        assert np.array_equal(canonical(g.bonds()), canonical(bonds_of_oracle(o)))
        assert np.array_equal(g.states(), o.state)
        assert n_a < 10 or len(g.bonds()) > n_a // 10
