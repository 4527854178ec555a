"""The constraint-graph path's parallel pass, resolve and continuation at the
sizes where they change course: more events than the 32 a warp keeps on its
lanes, runs that come round the box to disks they moved, dense chains whose
components fail to continue, meet and merge, and launches of several legs that
begin the next leg without a barrier of its own. Bit-exact against the oracle,
as everywhere on this path."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2004_11040_gb300 import ecmc, synth

from test_gpu_graph import assert_graph_parity

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,k,ell,legs", [
    (48, 6, 1.7, 3),    # about 31 to 33 events a chain and leg: one flush or two
    (48, 5, 3.6, 2),    # 66 events: three flushes, the row of 48 disks passed once
    (12, 3, 2.5, 3),    # several laps of a row of 12 in a leg
    (6, 1, 9.0, 2),     # one chain, ell beyond the box side
    (5, 25, 0.8, 2),    # every disk active
])
def test_long_runs_and_laps(m, k, ell, legs):
    assert_graph_parity(synth.lattice_start(m, 0.70, k, seed=m + k), ell, legs)


@pytest.mark.parametrize("n,k,ell,legs,windows", [
    (300, 30, 1.0, 24, 1),
    (300, 60, 2.0, 10, 1),
    (500, 20, 1.5, 10, 3),
])
def test_dense_two_dimensional_chains_over_many_legs(n, k, ell, legs, windows):
    """Cross-row liftings with many chains: failed continuations, takeovers and
    merged components in most legs."""
    _, st = assert_graph_parity(synth.rsa_start(n, 0.5, k, seed=n + k), ell, legs, windows)
    assert st["repaired_chains"] > st["continued_chains"] > 0


@pytest.mark.parametrize("seed", [1, 2])
def test_staggered_pairs_many_legs(seed):
    s = synth.staggered_start(24, 0.5, 60, seed, row_shift=0.05, pair_shift=0.15)
    assert_graph_parity(s, 1.0, 16)


def test_budget_decisions_of_a_long_run():
    """With a liftings budget every block decides alike after each leg when the
    launch ends: many short runs, each against the same legs without a budget."""
    s = synth.lattice_start(40, 0.70, 40, seed=9)
    a = ecmc.System(s.x, s.y, s.active, s.box, 1.0, graph=True)
    b = ecmc.System(s.x, s.y, s.active, s.box, 1.0, graph=True)
    for q in range(40):
        fa, na = a.run(1 << 18, event_budget=1000 + 97 * q)
        fb, nb = b.run(na)
        assert na == nb and np.array_equal(fa, fb)
    for u, v in zip(a.positions(), b.positions()):
        assert np.array_equal(u, v)
    assert a.stats()["liftings"] == b.stats()["liftings"]
    a.close()
    b.close()


def test_record_limit_is_reported_only_if_a_chain_needs_it():
    """A run alone longer than the records of a chain goes on in the repair,
    which reports the shortage; with room for every event there is none."""
    s = synth.lattice_start(40, 0.70, 2, seed=3)
    last, legs = O.run_legs(s.x, s.y, s.active, s.box, 1.0, 1, search=2)
    most = int(np.bincount(legs[0].log["c"]).max()) + 1  # liftings and the stall
    ok = ecmc.System(s.x, s.y, s.active, s.box, 1.0, graph=True, undo_cap=most)
    ok.run(1)
    assert np.array_equal(ok.positions()[0], last.x)
    ok.close()
    short = ecmc.System(s.x, s.y, s.active, s.box, 1.0, graph=True, undo_cap=most - 2)
    with pytest.raises(ecmc.EcmcError) as e:
        short.run(1)
    assert e.value.code == ecmc.ECMC_ECAPACITY
    short.close()
