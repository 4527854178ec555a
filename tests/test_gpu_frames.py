"""Cell-scan contexts whose frames change kind: a lattice's rows out of reach of
each other run the row pass on the cells; turned around after some legs the
frame is general (its legs run along the arrows of the constraint graph, the
flag still on cells), and turned back it may be rows again. Flags, positions,
local times, active disks and the log against the oracle, which knows one way
only; and batches of contexts of both kinds. Bit-exact."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2004_11040_gb300 import ecmc, synth

from test_gpu_parity import assert_parity, chain_order

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,k,legs,turns,windows,aligned", [
    (40, 30, 3, 5, 1, True),
    (53, 20, 2, 4, 1, False),
    (40, 60, 2, 4, 3, True),
])
def test_frames_change_kind(m, k, legs, turns, windows, aligned):
    s = synth.lattice_start(m, 0.66, k, seed=m + k)
    nc = m if aligned else O.default_cells(s.box)
    sysm = ecmc.System(s.x, s.y, s.active, s.box, 1.0, cells_per_side=nc, windows=windows, log=True)
    x, y, act = s.x.copy(), s.y.copy(), s.active.copy()
    logs, rows = [], 0
    for turn in range(turns):
        sysm.set_direction(turn % 2)
        f, done = sysm.run(legs)
        assert done == legs
        a, b = (x, y) if turn % 2 == 0 else (y, x)
        last, per = O.run_legs(a, b, act, s.box, 1.0, legs, nc=nc, windows=windows)
        act = last.active
        if turn % 2 == 0:
            x = last.x
        else:
            y = last.x
        gx, gy, gt, ga = sysm.positions()
        assert np.array_equal(gx, x) and np.array_equal(gy, y) and np.array_equal(ga, act), turn
        assert np.array_equal(gt, last.t), turn
        assert f.tolist() == [r.flag for r in per], turn
        for q, r in enumerate(per):
            lg = r.log.copy()
            lg["leg"] = turn * legs + q
            logs.append(lg)
        if turn == 0:
            rows = sysm.stats()["row_windows"]
    st = sysm.stats()
    glog = chain_order(sysm.liftings())
    olog = chain_order(np.concatenate(logs))
    assert len(glog) == len(olog)
    for name in ("leg", "c", "i", "j", "t", "tau", "xi", "xj"):
        assert np.array_equal(glog[name], olog[name]), name
    assert rows == (legs * windows if aligned else 0)
    assert st["row_windows"] < turns * legs * windows  # a turned frame is general
    sysm.close()


def test_batch_of_row_and_general_contexts():
    starts = [synth.lattice_start(40, 0.70, 16, seed=1), synth.rsa_start(400, 0.45, 8, seed=2),
              synth.lattice_start(44, 0.66, 20, seed=3)]
    mk = lambda: [ecmc.System(s.x, s.y, s.active, s.box, 1.0, cells_per_side=s.m) for s in starts]
    both, alone = mk(), mk()
    b = ecmc.ecmc_batch_create()
    budgets = [900, 200, 0]
    lifts, legs, ms = ecmc.ecmc_batch_run(b, [q.ctx for q in both], 12, budgets)
    assert ms > 0 and legs[2] == 12 and (lifts[:2] >= budgets[:2]).all()
    for q, s in enumerate(alone):
        s.run(int(legs[q]))
        assert s.stats()["liftings"] == lifts[q]
        for u, v in zip(both[q].positions(), s.positions()):
            assert np.array_equal(u, v)
    ecmc.ecmc_batch_destroy(b)
    for s in both + alone:
        s.close()


@pytest.mark.parametrize("n,k,windows,nc8", [(400, 60, 1, False), (400, 60, 4, False),
                                             (300, 20, 1, True)])
def test_general_frames_dense_flags_on_cells(n, k, windows, nc8):
    s = synth.rsa_start(n, 0.5, k, seed=n + k)
    nc = int(s.box / 1.55) if nc8 else 0  # 8 slots per cell
    assert_parity(s, 1.2, 6, nc=nc, windows=windows)
