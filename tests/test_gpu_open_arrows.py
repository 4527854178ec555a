"""A large frame's first launch of few legs, and the leg without allocation, run
with arrows that were searched for the near columns only. Boxes so sparse that disks come to where such an arrow ends
(the launch is then done again with the arrows completed), dense ones where none
does, small boxes (never so, but for the leg without allocation), the launches
after the first and turns: against the oracle, bit for bit.
"""
import math
from types import SimpleNamespace

import numpy as np
import pytest

from oracle import oracle as O
from paper_2004_11040_gb300 import ecmc
from test_gpu_far_arrows import hexagonal, sparse

pytestmark = pytest.mark.gpu


def box(kind, n, size, k):
    s = hexagonal(n, size, n) if kind == "hex" else sparse(n, size, n)
    rng = np.random.default_rng(n + k)
    s.active = rng.choice(s.n, min(k, s.n), replace=False).astype(np.int32)
    return s


def legs_of(x, y, active, s, ell, legs, nc):
    return O.run_legs(x, y, active, s.box, ell, legs, d=1.0, nc=nc, search=1)


# sparse boxes of 4 to 60 disks, up to 17 to 65 columns; rows of disks with few
# arrows to the rows beside
CASES = [("sparse", 4, 17.0, 1), ("sparse", 12, 41.3, 3), ("sparse", 40, 41.3, 8),
         ("sparse", 60, 65.7, 60), ("hex", 420, 0.60, 12), ("hex", 900, 0.62, 200),
         ("hex", 900, 0.60, 4)]


LARGE = [("hex", 140000, 0.012, 32), ("hex", 140000, 0.60, 64)]


@pytest.mark.parametrize("kind,n,size,k,ell,legs", [
    (*c, ell, legs) for c in CASES for ell, legs in [(1.0, 8), (2.0, 4), (1.0, 2)]] + [
    (*c, ell, legs) for c in LARGE for ell, legs in [(1.0, 8), (2.0, 4), (0.3, 2)]])
def test_first_launches_equal_oracle(kind, n, size, k, ell, legs):
    s = box(kind, n, size, k)
    nc = O.default_cells(s.box, 1.0)
    q = ecmc.System(s.x, s.y, s.active, s.box, ell, log=True)
    x, y, a, log = s.x, s.y, s.active, []
    for turn in (0, 1) if n > 100000 else (0, 1, 0):
        q.set_direction(turn)
        for part in (legs, 3):  # the frame's first launch, and one after it
            flags, done = q.run(part)
            u, v = (y, x) if turn else (x, y)
            last, runs = legs_of(u, v, a, s, ell, part, nc)
            x, y = (v, last.x) if turn else (last.x, v)
            a = last.active
            log += [len(r.log) for r in runs]
            assert done == part and list(flags) == [r.flag for r in runs]
            gx, gy, gt, ga = q.positions()
            assert np.array_equal(gx, x) and np.array_equal(gy, y)
            assert np.array_equal(gt, last.t) and np.array_equal(ga, a)
    st = q.stats()
    got = q.liftings()
    q.close()
    assert st["liftings"] == sum(log) == len(got) and st["legs"] == len(log)
    assert [int((got["leg"] == g).sum()) for g in range(len(log))] == log
    assert st["order_errors"] == 0 and st["horizon_asserts"] == 0


@pytest.mark.parametrize("ell", [1.0, 7.5])
@pytest.mark.parametrize("kind,n,size,k", CASES)
def test_leg_without_allocation(kind, n, size, k, ell):
    import torch
    s = box(kind, n, size, k)
    nc = O.default_cells(s.box, 1.0)
    last, runs = legs_of(s.x, s.y, s.active, s, ell, 1, nc)
    x, y = torch.from_numpy(s.x).cuda(), torch.from_numpy(s.y).cuda()
    a, t = torch.from_numpy(s.active).cuda(), torch.empty(s.n, dtype=torch.float64, device="cuda")
    flag, lifts = ecmc.ecmc_leg_noalloc(s.n, s.box, 1.0, ell, len(s.active), 0, x, y, a, t)
    assert np.array_equal(x.cpu().numpy(), last.x) and np.array_equal(t.cpu().numpy(), last.t)
    assert np.array_equal(a.cpu().numpy(), last.active)
    assert flag == runs[0].flag and lifts == len(runs[0].log)


@pytest.mark.parametrize("case", [("sparse", 40, 41.3, 8), LARGE[0]])
def test_budgets_batches_and_long_launches(case):
    s = box(*case)
    nc = O.default_cells(s.box, 1.0)
    last, runs = legs_of(s.x, s.y, s.active, s, 1.0, 30, nc)
    alone, long_, batched = [ecmc.System(s.x, s.y, s.active, s.box, 1.0) for _ in range(3)]
    budget = sum(len(r.log) for r in runs[:5])
    flags, done = alone.run(8, event_budget=max(1, budget))
    assert done <= 8
    while done < 30:
        done += alone.run(min(4, 30 - done))[1]
    long_.run(30)
    other = ecmc.System(s.x, s.y, s.active, s.box, 1.0)
    b = ecmc.ecmc_batch_create()
    ecmc.ecmc_batch_run(b, [batched.ctx, other.ctx], 8)
    ecmc.ecmc_batch_run(b, [batched.ctx], 22)
    ecmc.ecmc_batch_destroy(b)
    for q in (alone, long_, batched):
        x, _, t, a = q.positions()
        assert np.array_equal(x, last.x) and np.array_equal(t, last.t)
        assert np.array_equal(a, last.active)
        assert q.stats()["liftings"] == sum(len(r.log) for r in runs)
        q.close()
    other.close()
