"""Coordinates of -0.0 lie in [0, L): frames of rings, general frames, both kinds
of context, both directions and the leg that allocates nothing give what they
give for 0.0, and what the oracle gives. Tolerance: bit-exact (0.0 == -0.0).
"""
import os
import re
from types import SimpleNamespace

import numpy as np
import pytest

from oracle import oracle as O
from paper_2004_11040_gb300 import ecmc, synth

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2004_11040_gb300", "csrc")


def test_the_build_orders_no_coordinate_as_given():
    """The build ranks coordinates by their bits, where -0.0 is the largest of
    all: every read of an input coordinate takes it through coord()."""
    text = open(os.path.join(CSRC, "graph.cu")).read()
    reads = re.findall(r"(\w*\(?)b\.[xy]\[", text)
    assert len(reads) >= 8 and set(reads) == {"coord("}, reads


def ring_box(short_last):
    """24 rows of cells (side 1.35 d), each a ring; every row has a disk at x = 0
    and row 0 two at y = 0. The last row may hold fewer disks than a cell has
    slots."""
    rng = np.random.default_rng(7)
    nc, a, w = 24, 1.35, 0.25
    box = nc * a
    x, y = [], []
    for r in range(nc):
        m = 2 if short_last and r == nc - 1 else int(rng.integers(3, 25))
        gaps = rng.random(m)
        gaps *= (box - m) / gaps.sum()
        row = np.cumsum(1.0 + gaps)
        x.append((row - row[rng.integers(m)]) % box)
        y.append(r * a + 1e-3 + w * rng.random(m))
        if r == 0:
            y[-1][:2] = 0.0
    x, y = np.concatenate(x), np.concatenate(y)
    x[x >= box] = 0.0
    p = rng.permutation(len(x))
    active = rng.choice(len(x), size=30, replace=False).astype(np.int32)
    return SimpleNamespace(x=x[p], y=y[p], active=active, box=box, d=1.0, k=30), nc


def general_box():
    """A random packing moved so that one disk lies at x = 0 and another at y = 0."""
    s = synth.rsa_start(400, 0.45, 25, seed=11)
    x, y = (s.x - s.x[17]) % s.box, (s.y - s.y[230]) % s.box
    x[x >= s.box] = 0.0
    y[y >= s.box] = 0.0
    start = SimpleNamespace(x=x, y=y, active=s.active, box=s.box, d=s.d, k=25)
    return start, O.default_cells(s.box, s.d)


BOXES = {"rings": lambda: ring_box(False), "rings_short_last": lambda: ring_box(True),
         "general": general_box}


def negated(s):
    neg = lambda v: np.where(v == 0.0, -0.0, v)
    out = SimpleNamespace(**{**vars(s), "x": neg(s.x), "y": neg(s.y)})
    assert np.signbit(out.x).any() and np.signbit(out.y).any()
    return out


def sweep(s, nc, graph):
    q = ecmc.System(s.x, s.y, s.active, s.box, 1.0, d=s.d, cells_per_side=nc, graph=graph)
    out = []
    for direction in (0, 1, 0):
        q.set_direction(direction)
        flags, done = q.run(2)
        assert done == 2
        out += [flags, *q.positions()]
    rows = q.stats()["row_windows"]
    q.close()
    return out, rows


@pytest.mark.gpu
@pytest.mark.parametrize("graph", [False, True])
@pytest.mark.parametrize("box", sorted(BOXES))
def test_negative_zero_equals_zero(box, graph):
    s, nc = BOXES[box]()
    got, rows = sweep(negated(s), nc, graph)
    want, rows0 = sweep(s, nc, graph)
    assert rows == rows0 and (graph or box == "general" or rows > 0)
    for a, b in zip(got, want):
        assert np.array_equal(a, b)
    last, legs = O.run_legs(s.x, s.y, s.active, s.box, 1.0, 2, d=s.d, nc=nc,
                            search=2 if graph else 1)
    flags, x, y, t, active = got[:5]
    assert np.array_equal(x, last.x) and np.array_equal(y, s.y) and np.array_equal(t, last.t)
    assert np.array_equal(active, last.active)
    assert list(flags) == [r.flag for r in legs]


@pytest.mark.gpu
@pytest.mark.parametrize("box", sorted(BOXES))
def test_negative_zero_without_allocation(box):
    import torch
    s, nc = BOXES[box]()
    last, legs = O.run_legs(s.x, s.y, s.active, s.box, 1.0, 1, d=s.d, nc=nc, search=1)
    z = negated(s)
    x, y = torch.from_numpy(z.x).cuda(), torch.from_numpy(z.y).cuda()
    active = torch.from_numpy(s.active).cuda()
    t = torch.empty_like(x)
    flag, lifts = ecmc.ecmc_leg_noalloc(len(s.x), s.box, s.d, 1.0, s.k, nc, x, y, active, t)
    assert np.array_equal(x.cpu().numpy(), last.x) and np.array_equal(t.cpu().numpy(), last.t)
    assert np.array_equal(active.cpu().numpy(), last.active)
    assert flag == legs[0].flag and lifts == len(legs[0].log)
