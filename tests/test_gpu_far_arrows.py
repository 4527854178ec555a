"""Arrows to disks many columns ahead. Rows of disks little less than d apart in
y give few disks an arrow to the rows beside, most of them far along the row:
the build's search by blocks of columns, at the edges of the blocks and of the
box, against the definition (all pairs), in both directions; and its time
against a build whose arrows all are near. Tolerance: bit-exact.
"""
import math
import time
from types import SimpleNamespace

import numpy as np
import pytest

from oracle import oracle as O
from paper_2004_11040_gb300 import ecmc, synth

pytestmark = pytest.mark.gpu


def hexagonal(n, eta, seed, k=4):
    """About n disks (d = 1) on a triangular lattice, each displaced inside the
    circle that keeps it clear of its neighbours."""
    rows = max(4, 2 * round(math.sqrt(n * 2.0 / math.sqrt(3.0)) / 2.0))
    cols = max(4, round(n / rows))
    n = rows * cols
    box = math.sqrt(n * math.pi / (4.0 * eta))
    sx, sy = box / cols, box / rows
    reach = 0.49 * (min(sx, math.hypot(0.5 * sx, sy)) - 1.0)
    rng = np.random.default_rng(seed)
    r, phi = reach * np.sqrt(rng.random(n)), 2.0 * math.pi * rng.random(n)
    i, j = np.arange(n) % cols, np.arange(n) // cols
    x = np.mod((i + 0.25 + 0.5 * (j % 2)) * sx + r * np.cos(phi), box)
    y = np.mod((j + 0.5) * sy + r * np.sin(phi), box)
    p = rng.permutation(n)
    active = rng.choice(n, k, replace=False).astype(np.int32)
    return SimpleNamespace(x=x[p], y=y[p], active=active, box=box, d=1.0, n=n)


def sparse(n, box, seed, grid=0.0):
    """n disks at random, on a grid of that step if there is one: equal times of
    flight, disks d or d/2 apart in y."""
    rng = np.random.default_rng(seed)
    x, y = [], []
    while len(x) < n:
        u, v = rng.random(2) * box
        if grid:
            u, v = grid * int(u / grid), grid * int(v / grid)
        if all(math.hypot(min(abs(u - p), box - abs(u - p)),
                          min(abs(v - q), box - abs(v - q))) >= 1.0 for p, q in zip(x, y)):
            x.append(u)
            y.append(v)
    return SimpleNamespace(x=np.array(x), y=np.array(y), active=np.arange(2, dtype=np.int32),
                           box=box, d=1.0, n=n)


# boxes of 8, 9, 10, 15, 16, 17, 23, 24, 25, 33 and more columns; a few disks in many
CASES = [("hex", n, eta) for n, eta in [(60, 0.66), (64, 0.62), (72, 0.60), (180, 0.62),
                                        (196, 0.60), (224, 0.60), (420, 0.62), (460, 0.62),
                                        (484, 0.62), (900, 0.60), (900, 0.66), (2000, 0.58)]] + \
        [("sparse", n, box) for n, box in [(3, 9.5), (5, 17.0), (12, 41.3), (40, 64.9)]] + \
        [("grid", n, box) for n, box in [(20, 9.5), (40, 17.0), (150, 24.0), (60, 40.0)]]


@pytest.mark.parametrize("wide", [False, True])
@pytest.mark.parametrize("kind,n,size", CASES)
def test_far_arrows_equal_the_definition(kind, n, size, wide):
    s = hexagonal(n, size, n) if kind == "hex" else sparse(n, size, n, 0.25 * (kind == "grid"))
    nc = math.ceil(s.box / 1.6) if wide else 0  # cells of eight slots, or of four
    q = ecmc.System(s.x, s.y, s.active, s.box, 1.0, cells_per_side=nc, graph=True)
    a, _ = q.arrows()
    assert np.array_equal(a, O.graph3(s.x, s.y, s.box, d=1.0, search=0))
    q.set_direction(1)
    a, _ = q.arrows()
    q.close()
    assert np.array_equal(a, O.graph3(s.y, s.x, s.box, d=1.0, search=0))


def test_far_arrows_cost_little_more_than_near_ones():
    """(859 us against 111 when each far search went over the whole row.)"""
    def us(s):
        q = ecmc.System(s.x, s.y, s.active, s.box, 1.0)
        best = math.inf
        for r in range(12):
            t = time.perf_counter()
            q.set_direction(1 - r % 2)
            q.set_direction(r % 2)
            best = min(best, 0.5e6 * (time.perf_counter() - t))
        q.close()
        return best

    far = us(hexagonal(360000, 0.60, 1, k=16))
    near = us(synth.lattice_start(600, 0.60, 16, 1))
    assert far < 3.0 * near, (far, near)
