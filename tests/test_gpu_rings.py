"""Frames of rings (every cell row a row of disks out of reach of the others):
rings of every length around a warp's stretch of 31 events, legs that need
several stretches or come round the ring, against the oracle, bit for bit.

A ring frame needs each row within 0.86 d in y and d or more from the rows
beside; a frame one of whose rows is wider runs along the arrows of G(3).
Tolerance: bit-exact (positions, local times, liftings, flags).
"""
from types import SimpleNamespace

import numpy as np
import pytest

from test_gpu_rowpass import oracle, run, same

pytestmark = pytest.mark.gpu


def rings(nc, a, spread, lengths, k, seed, wide_row=False):
    """nc rows of cells of side a (d = 1), row r with lengths[r mod ..] disks
    spread along x with random gaps; ids shuffled over the box."""
    rng = np.random.default_rng(seed)
    box = nc * a
    x, y = [], []
    for r in range(nc):
        m = lengths[r % len(lengths)]
        gaps = rng.random(m)
        gaps *= (box - m) / gaps.sum()
        x.append((rng.random() * box + np.cumsum(1.0 + gaps)) % box)
        w = spread if not (wide_row and r == nc // 2) else 0.9
        lo = (r + 0.5) * a - 0.5 * w
        y.append(lo + w * rng.random(m))
        if m > 1:  # the row's whole width is taken
            y[-1][0], y[-1][1] = lo, lo + w
    x, y = np.concatenate(x), np.concatenate(y)
    p = rng.permutation(len(x))
    active = rng.choice(len(x), size=min(k, len(x)), replace=False).astype(np.int32)
    return SimpleNamespace(x=x[p], y=y[p], active=active, box=box, d=1.0, k=len(active))


EDGES = [1, 2, 3, 30, 31, 32, 33, 5, 16]
LONG = [62, 63, 64, 65, 40, 1]


@pytest.mark.parametrize("nc,a,spread,lengths,k,ell,windows,seed", [
    (40, 1.35, 0.3, EDGES, 1, 1.0, 1, 1),
    (40, 1.35, 0.3, EDGES, 40, 0.05, 1, 2),    # legs of one event or two
    (40, 1.35, 0.3, EDGES, 60, 1.0, 1, 3),
    (40, 1.35, 0.3, EDGES, 300, 3.0, 1, 4),    # short rings come round
    (48, 1.6, 0.55, LONG, 24, 2.0, 1, 5),      # cells of eight slots
    (48, 1.6, 0.55, LONG, 48, 6.0, 1, 6),      # several stretches
    (48, 1.6, 0.55, LONG, 200, 4.0, 3, 7),     # claim windows
])
def test_rings_equal_oracle(nc, a, spread, lengths, k, ell, windows, seed):
    s = rings(nc, a, spread, lengths, k, seed)
    g = run(s, ell, 4, windows, nc=nc)
    same(g, oracle(s, ell, 4, windows, nc=nc))
    assert 0 <= g[5]["row_windows"] <= 4 * windows
    if ell <= 0.05:
        assert g[5]["row_windows"] == 4 * windows


@pytest.mark.parametrize("k,ell,windows,seed", [
    (60, 1.0, 1, 3), (300, 3.0, 1, 4), (200, 2.0, 3, 7),
])
def test_rings_of_a_graph_context(k, ell, windows, seed):
    """With the arrows of G(3) a ring's successor may be any of the three."""
    s = rings(40, 1.35, 0.3, EDGES, k, seed)
    g = run(s, ell, 4, windows, graph=True, nc=40)
    same(g, oracle(s, ell, 4, windows, search=2, nc=40))


def test_a_wide_row_is_no_ring():
    s = rings(40, 1.6, 0.3, [10, 20, 3], 60, 8, wide_row=True)
    g = run(s, 1.0, 4, nc=40)
    same(g, oracle(s, 1.0, 4, nc=40))
    assert g[5]["row_windows"] == 0
