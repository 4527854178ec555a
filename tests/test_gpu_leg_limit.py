"""The legs of one call: a constraint-graph context refuses 2^24 legs x windows
(the header says so), nothing is run; a cell-scan context takes any number,
until its budget.
"""
import os

import numpy as np
import pytest

from paper_2004_11040_gb300 import ecmc, synth

HEADER = open(os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "include",
                           "ecmc.h")).read()


def test_the_header_states_the_limit():
    for call in ("n_legs", "max_legs"):
        assert f"EINVAL (with ECMC_GRAPH also {call} x windows >= 2^24)" in HEADER


@pytest.mark.gpu
@pytest.mark.parametrize("windows,legs", [(1, 1 << 24), (4096, 4096)])
def test_legs_of_one_call(windows, legs):
    s = synth.lattice_start(16, 0.70, 4, seed=1)
    graph = ecmc.System(s.x, s.y, s.active, s.box, 0.5, windows=windows, graph=True)
    with pytest.raises(ecmc.EcmcError) as e:
        ecmc.ecmc_run_to_breakpoint(graph.ctx, legs, 10)
    assert e.value.code == ecmc.ECMC_EINVAL
    batch = ecmc.ecmc_batch_create()
    with pytest.raises(ecmc.EcmcError) as e:
        ecmc.ecmc_batch_run(batch, [graph.ctx], legs, [10])
    assert e.value.code == ecmc.ECMC_EINVAL
    assert graph.stats()["legs"] == 0 and np.array_equal(graph.positions()[0], s.x)
    cells = ecmc.System(s.x, s.y, s.active, s.box, 0.5, windows=windows)
    done = ecmc.ecmc_run_to_breakpoint(cells.ctx, legs, 10)
    assert 0 < done < legs and cells.stats()["liftings"] >= 10
    ecmc.ecmc_batch_destroy(batch)
    graph.close()
    cells.close()
