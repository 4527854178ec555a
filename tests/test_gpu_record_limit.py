"""A chain that needs more event records than the context has (undo_cap) ends
the leg with ECAPACITY after the repair round that found it, also where more
than 64 chains would be merged into one component, and other systems of the
launch finish their leg.
"""
import functools
import time

import numpy as np
import pytest

from oracle import oracle as O
from paper_2004_11040_gb300 import ecmc, synth

pytestmark = pytest.mark.gpu


start = functools.lru_cache(None)(synth.rsa_start)


def system(s, undo_cap, graph):
    return ecmc.System(s.x, s.y, s.active, s.box, 1.0, d=s.d, undo_cap=undo_cap, graph=graph)


@pytest.mark.parametrize("graph", [False, True])
@pytest.mark.parametrize("n,k", [(900, 60), (900, 200), (900, 600)])
def test_out_of_records_ends_the_leg(n, k, graph):
    s = start(n, 0.48, k, seed=n + k)
    q = system(s, 2, graph)
    with pytest.raises(ecmc.EcmcError) as e:
        q.run(3)
    assert e.value.code == ecmc.ECMC_ECAPACITY
    # every chain enters the first round's repair at most once, or is taken in
    # by one component there; no round follows
    assert q.stats()["repaired_chains"] <= 2 * k
    q.close()


@pytest.mark.parametrize("graph", [False, True])
def test_other_systems_of_the_launch_finish(graph):
    short = start(900, 0.48, 200, seed=5)
    s = start(900, 0.48, 90, seed=6)
    systems = [system(short, 2, graph), system(s, 0, graph)]
    batch = ecmc.ecmc_batch_create()
    with pytest.raises(ecmc.EcmcError) as e:
        ecmc.ecmc_batch_run(batch, [q.ctx for q in systems], 1)
    assert e.value.code == ecmc.ECMC_ECAPACITY
    x, _, t, a = systems[1].positions()
    last, legs = O.run_legs(s.x, s.y, s.active, s.box, 1.0, 1, d=s.d,
                            nc=O.default_cells(s.box, s.d), search=2 if graph else 1)
    assert np.array_equal(x, last.x) and np.array_equal(t, last.t)
    assert np.array_equal(a, last.active)
    assert systems[1].stats()["liftings"] == len(legs[0].log)
    ecmc.ecmc_batch_destroy(batch)
    for q in systems:
        q.close()


def test_out_of_records_without_allocation():
    import torch
    s = synth.lattice_start(48, 0.70, 120, seed=4)
    x, y = torch.from_numpy(s.x).cuda(), torch.from_numpy(s.y).cuda()
    a, t = torch.from_numpy(s.active).cuda(), torch.empty(s.n, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    with pytest.raises(ecmc.EcmcError) as e:
        ecmc.ecmc_leg_noalloc(s.n, s.box, s.d, 25.0, s.k, 0, x, y, a, t)
    assert e.value.code == ecmc.ECMC_ECAPACITY
    assert time.perf_counter() - t0 < 5.0
    assert np.array_equal(x.cpu().numpy(), s.x) and np.array_equal(a.cpu().numpy(), s.active)
