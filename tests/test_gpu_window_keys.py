"""Claim windows use two sets of touch keys in turn: even and odd numbers of
windows, several legs (the next leg's first window takes up the first set
again), several systems in a launch, against the oracle, bit for bit.
"""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2004_11040_gb300 import batch, ecmc, synth

pytestmark = pytest.mark.gpu


def check(sysm, s, ell, legs, windows, search):
    last, runs = O.run_legs(s.x, s.y, s.active, s.box, ell, legs, d=s.d,
                            nc=O.default_cells(s.box, s.d), windows=windows, search=search)
    x, _, t, a = sysm.positions()
    assert np.array_equal(x, last.x) and np.array_equal(t, last.t)
    assert np.array_equal(a, last.active)
    st = sysm.stats()
    assert st["liftings"] == sum(len(r.log) for r in runs)
    assert st["conflict_windows"] == sum(int(r.wflags.sum()) for r in runs)
    assert st["order_errors"] == 0 and st["horizon_asserts"] == 0
    return np.array([r.flag for r in runs], dtype=np.uint8)


@pytest.mark.parametrize("graph", [False, True])
@pytest.mark.parametrize("windows", [2, 3, 4, 7])
def test_windows_equal_oracle(windows, graph):
    s = synth.rsa_start(600, 0.47, 120, seed=windows)
    sysm = ecmc.System(s.x, s.y, s.active, s.box, 1.5, d=s.d, windows=windows, graph=graph)
    flags = np.concatenate([sysm.run(3)[0], sysm.run(2)[0]])
    assert np.array_equal(flags, check(sysm, s, 1.5, 5, windows, 2 if graph else 1))
    sysm.close()


@pytest.mark.parametrize("windows", [2, 5])
def test_windows_of_several_systems(windows):
    starts = [synth.rsa_start(400, 0.45, 20 + 30 * q, seed=q) for q in range(3)]
    systems = [ecmc.System(s.x, s.y, s.active, s.box, 1.0, d=s.d, windows=windows)
               for s in starts]
    b = ecmc.ecmc_batch_create()
    ecmc.ecmc_batch_run(b, [q.ctx for q in systems], 4)
    ecmc.ecmc_batch_destroy(b)
    for s, q in zip(starts, systems):
        check(q, s, 1.0, 4, windows, 1)
        q.close()
