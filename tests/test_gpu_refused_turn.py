"""A direction change that is refused (disks that overlapped at the start have
left a cell with more of them than it has slots) leaves the context as it was:
positions, and the legs that follow.
"""
from types import SimpleNamespace

import numpy as np
import pytest

from paper_2004_11040_gb300 import ecmc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("graph", [False, True])
def test_refused_direction_change(graph):
    # four disks in one cell (side 1.25 d); the active one stops at contact in
    # the same cell, and what is left of the leg moves the last of the four 0.01
    x = np.array([6.20, 6.21, 6.22, 6.23, 3.9, 1.3, 8.6, 2.5])
    y = np.array([5.60, 5.60, 5.60, 5.60, 5.6, 1.9, 2.0, 8.8])
    s = SimpleNamespace(x=x, y=y, active=np.array([4], dtype=np.int32), box=10.0)

    def system():
        q = ecmc.System(s.x, s.y, s.active, s.box, 1.31, cells_per_side=8, graph=graph)
        q.run(1)
        return q

    a, b = system(), system()
    before = a.positions()
    assert before[0][4] == pytest.approx(5.2) and before[3][0] != 4
    with pytest.raises(ecmc.EcmcError) as e:
        a.set_direction(1)
    assert e.value.code == ecmc.ECMC_ECAPACITY
    for p, q in zip(a.positions(), before):
        assert np.array_equal(p, q)
    for q in (a, b):
        q.run(3)
    for p, q in zip(a.positions(), b.positions()):
        assert np.array_equal(p, q)
    a.close()
    b.close()
