"""What a context is planned to hold (no GPU): a context that will never run
along rings holds no places of rings."""
from paper_2004_11040_gb300 import ecmc


def planned(flags, ell=1.0, n=65536, box=256.0):
    p = ecmc.ecmc_params(n, box, 0.95, ell, 256, 256, flags, 0, 0, 1, 0)
    return ecmc.ecmc_context_bytes(p)


def test_no_places_without_rings():
    n = 65536
    assert planned(ecmc.ECMC_NO_ROWPASS) <= planned(0) - 16 * n
    # a leg as long as the box never runs along rings either
    assert planned(0, ell=256.0) <= planned(0) - 16 * n
