"""The leg that allocates nothing over every kind of frame and at its limits:
rings, general frames, cells of four and of eight slots, against the oracle,
bit for bit; and the refusals of sizes and inputs.
"""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2004_11040_gb300 import ecmc, synth

pytestmark = pytest.mark.gpu


def leg(s, ell, nc=0):
    import torch
    x = torch.tensor(s.x, dtype=torch.float64, device="cuda")
    y = torch.tensor(s.y, dtype=torch.float64, device="cuda")
    act = torch.tensor(s.active, dtype=torch.int32, device="cuda")
    t = torch.empty_like(x)
    flag, lifts = ecmc.ecmc_leg_noalloc(len(s.x), s.box, s.d, ell, len(s.active), nc, x, y, act, t)
    return flag, lifts, x.cpu().numpy(), t.cpu().numpy(), act.cpu().numpy()


@pytest.mark.parametrize("kind,n,k,ell,cells", [
    ("lattice", 32, 1, 0.5, "default"), ("lattice", 32, 60, 1.0, "lattice"),
    ("lattice", 32, 6, 8.0, "lattice"),   # a leg that comes round its ring
    ("rsa", 3, 1, 0.5, "default"), ("rsa", 900, 40, 1.0, "default"),
    ("rsa", 900, 200, 1.0, "wide"), ("staggered", 24, 50, 1.0, "default"),
])
def test_noalloc_equals_oracle(kind, n, k, ell, cells):
    if kind == "rsa":
        s = synth.rsa_start(n, 0.45 if n > 3 else 0.15, k, seed=n + k)
    elif kind == "lattice":
        s = synth.lattice_start(n, 0.66, k, seed=n + k)
    else:
        s = synth.staggered_start(n, 0.5, k, seed=3, row_shift=0.05, pair_shift=0.15)
    nc = O.default_cells(s.box, s.d)
    nc = {"default": nc, "lattice": n, "wide": int(s.box / (1.5 * s.d))}[cells]
    flag, lifts, x, t, act = leg(s, ell, nc)
    last, legs = O.run_legs(s.x, s.y, s.active, s.box, ell, 1, d=s.d, nc=nc, search=1)
    assert np.array_equal(x, last.x) and np.array_equal(t, last.t)
    assert np.array_equal(act, last.active)
    assert flag == legs[0].flag and lifts == len(legs[0].log)


def test_noalloc_refusals():
    import torch
    s = synth.lattice_start(32, 0.70, 12, seed=4)
    x = torch.tensor(s.x, dtype=torch.float64, device="cuda")
    y = torch.tensor(s.y, dtype=torch.float64, device="cuda")
    act = torch.tensor(s.active, dtype=torch.int32, device="cuda")
    t = torch.empty_like(x)

    def code(n=s.n, box=s.box, ell=1.0, k=s.k, x=x, y=y, act=act):
        with pytest.raises(ecmc.EcmcError) as e:
            ecmc.ecmc_leg_noalloc(n, box, s.d, ell, k, 0, x, y, act, t)
        return e.value.code

    bad_x = x.clone()
    bad_x[5] = float("nan")
    bad_y = y.clone()
    bad_y[7] = s.box
    twice = act.clone()
    twice[3] = twice[2]
    beyond = act.clone()
    beyond[0] = s.n
    for kw in (dict(x=bad_x), dict(y=bad_y), dict(act=twice), dict(act=beyond)):
        assert code(**kw) == ecmc.ECMC_EINVAL
    assert code(ell=25.0) == ecmc.ECMC_ECAPACITY  # more events than a chain's records
    # more disks than slots
    m = 200_000
    small = torch.rand(m, dtype=torch.float64, device="cuda") * 30.0
    ids = torch.arange(2, dtype=torch.int32, device="cuda")
    t = torch.empty_like(small)
    assert code(n=m, box=32.0, k=2, x=small, y=small, act=ids) == ecmc.ECMC_ECAPACITY
    ids[1] = 0
    assert code(n=m, box=32.0, k=2, x=small, y=small, act=ids) == ecmc.ECMC_EINVAL
    # the inputs that were refused are as they were
    assert np.array_equal(x.cpu().numpy(), s.x) and np.array_equal(act.cpu().numpy(), s.active)
