"""The array behind ecmc_leg_noalloc holds what every accepted leg needs: the
sizes are accepted by a count of their own (ECMC_NOALLOC_SCRATCH_MIB), the leg's
arrays are laid out by graph_leg_bytes. No GPU is used.
"""
import ctypes as C
import math
import os
import re

import numpy as np
import pytest

from paper_2004_11040_gb300 import ecmc

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
HEADER = open(os.path.join(ROOT, "include", "ecmc.h")).read()
SOURCE = open(os.path.join(ROOT, "paper_2004_11040_gb300", "csrc", "ecmc.cu")).read()
ACCEPT = int(re.search(r"#define ECMC_NOALLOC_SCRATCH_MIB (\d+)", HEADER).group(1)) << 20
RECORDS = int(re.search(r"#define ECMC_NOALLOC_RECORDS (\d+)", HEADER).group(1))
ARRAY = int(re.search(r"NOALLOC_SCRATCH_BYTES = \(size_t\)(\d+) << 20", SOURCE).group(1)) << 20


def count(nslot, ncell, n, k):
    """The documented count: 33 bytes a slot, 4 a disk, 24.7 KB a chain, in parts
    on 256-byte boundaries."""
    parts = 3 * [8 * nslot] + 2 * [4 * nslot] + [4 * ncell, 4 * n] + 8 * [8 * k] + 22 * [4 * k]
    parts += [4 * (k + 1)] + 3 * [152] + [96 * RECORDS * k]
    off = 0
    for p in parts:
        off = (off + 255) // 256 * 256 + p
    return off


@pytest.fixture(scope="module")
def need():
    lib = ecmc.load()
    f = lib._Z15graph_leg_bytesPK11ecmc_paramsi
    f.restype, f.argtypes = C.c_size_t, [C.POINTER(ecmc.ecmc_params), C.c_int]
    return lambda n, box, k, nc: f(C.byref(ecmc.ecmc_params(n, box, 1.0, 1.0, k, nc, 0, RECORDS, 0,
                                                            1, 0)), nc)


@pytest.mark.parametrize("side,slots", [(1.00001, 4), (1.2, 4), (1.414, 4), (1.4143, 8), (1.66, 8)])
def test_accepted_sizes_fit(need, side, slots):
    most = 0
    for nc in sorted(set(np.geomspace(3, 600, 120).astype(int))):
        box = nc * side
        full = min(int(2.0 / math.sqrt(3.0) * box * box), nc * nc * slots)  # close packing
        for n in sorted({3, full // 3, 3 * full // 4, full}):
            if n < 3 or count(nc * nc * slots, nc * nc, n, 1) > ACCEPT:
                continue
            lo, hi = 1, n  # the largest accepted number of chains
            while lo < hi:
                mid = (lo + hi + 1) // 2
                if count(nc * nc * slots, nc * nc, n, mid) <= ACCEPT:
                    lo = mid
                else:
                    hi = mid - 1
            for k in {1, (lo + 1) // 2, lo}:
                most = max(most, need(n, box, k, nc))
    assert 0 < most <= ARRAY, (most, ARRAY)


def test_the_header_states_the_array():
    assert f"{ARRAY >> 20} MiB that the library" in re.sub(r"\s*\*\s*", " ", HEADER)
