"""Boxes whose cell rows hold so many particles that a tile's nine neighbour
rows have more than 65,535 staged entries: the forces of the FP64 mode, which
walks the same lists, against the oracle's."""
import numpy as np
import pytest

import oracle as orc
from helpers import force_errors
from test_gpu_boxes import P, gpu_from, lattice_box  # noqa: F401 (P is a fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sites", [2700, 4200])  # 67,632 and 105,132 staged entries
def test_forces(P, sites):  # noqa: F811
    L, x = lattice_box((sites, 5, 5), 41, jitter=0.1)
    n = len(x)
    o = orc.System(x, np.zeros((n, 3)), np.zeros(n, np.uint8), np.zeros(n, np.int8), cap=4)
    f_ref, e_ref = orc.forces(o, orc.MDParams(L=L, seed=41), use_cells=True)
    with gpu_from(P, L, o, 41, True) as g:
        f, e = g.forces()
        g.run(25)
        assert np.isfinite(g.positions()).all()
    err = force_errors(f, f_ref)
    assert err["max_over_rms"] < 1e-12, err
    assert e == pytest.approx(e_ref, rel=1e-12)
