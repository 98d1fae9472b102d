"""The list build's FP32 distance test, pinned on the CPU against FP64 (the
coordinates that the permutation writes and the test of a candidate from one of
the nine neighbour rows): with the widened radius no pair within the list radius
is lost, and the distance's error is no larger than that of coordinates in a
frame at the lower edges of a tile of rows."""
import math

import numpy as np

from test_decision_identities import build_coord, f32, fixed_point_constants, fma32, periodic_fx


def build_xyz(X, cell, L, nc):
    """x in the box (kept on the side of the cell that holds the bead), y and z
    from the lower edges of the bead's own row."""
    s = [f32(v / 4294967296.0) for v in L]
    x = np.float32(np.float32(X[0]) * s[0])
    if cell[0] == 0 and X[0] >= 0xC0000000:
        x = np.float32(x - f32(L[0]))
    if cell[0] == nc[0] - 1 and X[0] < 0x40000000:
        x = np.float32(x + f32(L[0]))
    out = [x]
    for k in (1, 2):
        inv = (1 << 64) // nc[k] + 1 if (1 << 64) % nc[k] else (1 << 64) // nc[k]
        ref = ((cell[k] << 32) * inv) >> 64
        d = (X[k] - ref) % (1 << 32)
        out.append(np.float32(np.float32(d - (1 << 32) if d >= 1 << 31 else d) * s[k]))
    return out


def r2_build(fi, fj, rows, img, L, nc):
    """The test's r^2: fj in the row `rows` = (dy, dz) away, x shifted for the image cell."""
    xj = np.float32(fj[0] + img * f32(L[0])) if img else fj[0]
    e = [np.float32(xj - fi[0])]
    for k in (1, 2):
        shifted = np.float32(fi[k] - np.float32(np.float32(rows[k - 1]) * f32(L[k] / nc[k])))
        e.append(np.float32(fj[k] - shifted))
    return fma32(e[2], e[2], fma32(e[1], e[1], np.float32(e[0] * e[0])))


def test_every_pair_within_the_list_radius_is_kept():
    rng = np.random.default_rng(74)
    rc, skin = 2.0 ** (1.0 / 6.0), 0.4
    rv = rc + skin
    for L in ((12.0, 12.0, 12.0), (107.24910150874837,) * 3, (5.28, 699.0, 5.28), (5.28, 1000.0, 1000.0), (1000.0,) * 3):
        nc = [int(math.floor(v / (rv * (1.0 + 1e-9)))) for v in L]
        rvb = rv * (1.0 + 1e-5) + 1e-6 * max(L)
        rv2_build = f32(rvb * rvb)
        Lfx_M = [fixed_point_constants(v) for v in L]
        worst = {"row": 0.0, "tile": 0.0}
        for _ in range(1200):
            xi = [float(rng.uniform(0, v)) for v in L]
            if rng.random() < 0.3:  # at a cell's edge
                k = int(rng.integers(0, 3))
                xi[k] = (int(rng.integers(0, nc[k])) * L[k] / nc[k] + float(rng.normal()) * 1e-7) % L[k]
            d = rng.normal(size=3)
            r = rv * (1.0 - float(rng.choice([rng.uniform(0, 1e-6), rng.uniform(0, 3e-3)])))
            xj = [(a + r * c / float(np.linalg.norm(d))) % v for a, c, v in zip(xi, d, L)]
            P = [[periodic_fx(v, *Lfx_M[k]) for k, v in enumerate(x)] for x in (xi, xj)]
            cells = [[(p[k] * nc[k]) >> 32 for k in range(3)] for p in P]
            rows = []
            for k in (1, 2):
                dc = cells[1][k] - cells[0][k]
                rows.append(dc - nc[k] if dc > 1 else dc + nc[k] if dc < -1 else dc)
            dx = cells[1][0] - cells[0][0]
            img = -1 if dx > 1 else 1 if dx < -1 else 0
            r2 = r2_build(build_xyz(P[0], cells[0], L, nc), build_xyz(P[1], cells[1], L, nc), rows, img, L, nc)
            assert r2 < rv2_build, (L, xi, xj, float(r2), float(rv2_build))
            # error against the exact distance of the two fixed-point positions, which both take
            ex = 0.0
            for k in range(3):
                q = (P[1][k] - P[0][k]) % (1 << 32)
                ex += ((q - (1 << 32) if q >= 1 << 31 else q) * (L[k] / 4294967296.0)) ** 2
            e = [np.float32(b - a) for a, b in zip(
                build_coord(*P[0], cells[0], (0, 0), 0, L, nc, cells[0][1], cells[0][2]),
                build_coord(*P[1], cells[1], rows, img, L, nc, cells[0][1], cells[0][2]))]
            tile = fma32(e[2], e[2], fma32(e[1], e[1], np.float32(e[0] * e[0])))
            worst["row"] = max(worst["row"], abs(math.sqrt(float(r2)) - math.sqrt(ex)))
            worst["tile"] = max(worst["tile"], abs(math.sqrt(float(tile)) - math.sqrt(ex)))
        # (one rounding more, of at most two edges, in each of y and z: half of 2.4e-7)
        assert worst["row"] <= worst["tile"] + 2.4e-7, (L, worst)
