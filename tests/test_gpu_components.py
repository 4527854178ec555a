"""Conflict components of every size, their member lists gathered from the
trees that the blocked chains' unions leave: single pairs, more than a warp's
buffer (32, 96 and 224 members), nearly every chain of the system, and several
systems in one launch. Against the oracle, bit for bit.
"""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2004_11040_gb300 import batch, ecmc, synth

pytestmark = pytest.mark.gpu


def expect(s, ell, legs, windows, search):
    nc = O.default_cells(s.box, s.d)
    return O.run_legs(s.x, s.y, s.active, s.box, ell, legs, d=s.d, nc=nc, windows=windows,
                      search=search)


@pytest.mark.parametrize("n,k,ell,windows", [
    (900, 2, 2.0, 1), (900, 90, 1.0, 1), (900, 220, 1.0, 1), (900, 220, 2.0, 2),
    (2500, 700, 1.0, 1), (2500, 900, 1.5, 1),
])
@pytest.mark.parametrize("graph", [True, False])
def test_components_equal_oracle(n, k, ell, windows, graph):
    s = synth.rsa_start(n, 0.48, k, seed=n + k)
    sysm = ecmc.System(s.x, s.y, s.active, s.box, ell, d=s.d, windows=windows, graph=graph)
    flags, done = sysm.run(3)
    x, _, t, a = sysm.positions()
    st = sysm.stats()
    sysm.close()
    last, legs = expect(s, ell, 3, windows, 2 if graph else 1)
    assert done == 3
    assert np.array_equal(flags, np.array([r.flag for r in legs], dtype=np.uint8))
    assert np.array_equal(x, last.x) and np.array_equal(t, last.t)
    assert np.array_equal(a, last.active)
    assert st["liftings"] == sum(len(r.log) for r in legs)
    assert st["order_errors"] == 0 and st["horizon_asserts"] == 0


def test_components_of_several_systems():
    starts = [synth.rsa_start(900, 0.48, k, seed=k) for k in (1, 220, 60, 300)]
    systems = [ecmc.System(s.x, s.y, s.active, s.box, 1.0, d=s.d) for s in starts]
    batch.run_batched(systems, 0, 3)
    for s, sysm in zip(starts, systems):
        x, _, t, a = sysm.positions()
        last, _ = expect(s, 1.0, 3, 1, 1)
        assert np.array_equal(x, last.x) and np.array_equal(t, last.t)
        assert np.array_equal(a, last.active)
        sysm.close()
