"""The autotuner's cache file: a choice stored under a key without the generation
of the kernels (files written before it was part of the key) is not taken; one
with it is, without a GPU."""
import numpy as np
import pytest


@pytest.fixture(scope="module")
def P():
    from paper_1409_7498_gb300 import build, polyrx
    build.build()
    return polyrx


KEY = "n=2048 rho=0.8500 cap=4 fp64=0 gamma=1 rx=0 rr=0 theta=0 k=0 steps=37|0.300000,|256x0x1,256x0x4,|1,"
CHOICE = "\t0.29999999999999999 256 0 1 4 0.0123\n"


def tune(P, path, n=2048):
    L = (n / 0.85) ** (1.0 / 3.0)
    x = np.random.default_rng(1).random((n, 3)) * L
    return P.prx_autotune(P.make_desc(n, L, adj_cap=4), x, None, np.zeros(n, np.uint8), np.zeros(n, np.int8), None,
                          steps=37, skins=(0.3,), shapes=((256, 0, 1), (256, 0, 4)), chunks=(1,), cache_path=str(path))


def test_older_choices_are_not_taken(P, tmp_path):
    path = tmp_path / "tune.txt"
    path.write_text(KEY + CHOICE)
    try:
        best, tried = tune(P, path)
    except P.PolyrxError:  # no GPU: none of the candidates can be timed
        return
    assert not best["cached"] and len(tried) == 4


def test_a_current_choice_is_taken(P, tmp_path):
    path = tmp_path / "tune.txt"
    path.write_text("g2 " + KEY.replace("n=2048", "n=2047") + CHOICE)  # (another key than the test above)
    best, tried = tune(P, path, 2047)
    assert best["cached"] and best["step_lanes"] == 4 and not tried
