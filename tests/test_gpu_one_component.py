"""Legs whose chains nearly all are one conflict component end as one component
of all chains, whose replay claims nothing: against the oracle, bit for bit.
"""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2004_11040_gb300 import ecmc, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("graph", [False, True])
@pytest.mark.parametrize("n,k,ell,windows", [(300, 66, 3.0, 1), (300, 150, 1.0, 1),
                                             (300, 290, 1.0, 1), (300, 200, 1.5, 2)])
def test_one_component_equals_oracle(n, k, ell, windows, graph):
    s = synth.rsa_start(n, 0.5, k, seed=n + k)
    q = ecmc.System(s.x, s.y, s.active, s.box, ell, d=s.d, windows=windows, graph=graph)
    flags, done = q.run(4)
    x, _, t, a = q.positions()
    st = q.stats()
    q.close()
    last, legs = O.run_legs(s.x, s.y, s.active, s.box, ell, 4, d=s.d,
                            nc=O.default_cells(s.box, s.d), windows=windows,
                            search=2 if graph else 1)
    assert done == 4 and list(flags) == [r.flag for r in legs]
    assert np.array_equal(x, last.x) and np.array_equal(t, last.t)
    assert np.array_equal(a, last.active)
    assert st["liftings"] == sum(len(r.log) for r in legs)
    assert st["order_errors"] == 0 and st["repaired_chains"] >= k
