"""The graph build's FP32 search keeps bounds of each time of flight: the exact
one (FP64, as the arrows are defined) lies between them, and the corridor they
are for is the exact one, for disks anywhere in boxes of any size and cells of
either kind. (Host emulation of the device's float operations; the device's
approximate square root is off by less than 2^-22, which the last assertion
leaves room for.)"""
import numpy as np
import pytest

f = np.float32


def in_cell(v, a, inv_a, nc):
    c = np.minimum(np.trunc(v * inv_a).astype(np.int64), nc - 1)
    r = v - c * a
    r32 = f(np.sign(r)) * f(np.abs(r)).astype(f)
    t = np.nextafter(r32, f(0), dtype=f)  # truncation toward zero at worst one ulp lower
    return c, np.where(np.abs(r32.astype(np.float64)) > np.abs(r), t, r32)


@pytest.mark.parametrize("nc,a,d", [(17, 1.0004, 1.0), (270, 1.01, 1.0), (2090, 1.45, 1.0),
                                    (64, 0.3705, 0.3701)])
def test_bounds_hold_the_exact_time_of_flight(nc, a, d):
    rng = np.random.default_rng(nc)
    L = nc * a
    n = 200000
    inv_a = nc / L
    a = L / nc
    xi, yi = rng.random(n) * L, rng.random(n) * L
    # a second disk up to 40 columns ahead and within 1.1 d in y, many near the edges
    # of the corridors
    dx = rng.random(n) * min(40.0 * a, 0.4 * L)
    dy = (2 * rng.random(n) - 1) * 1.1 * d
    near = rng.random(n)
    dy = np.where(near < 0.2, d * (1 - 10.0 ** rng.uniform(-9, -2, n)) * np.sign(dy), dy)
    dy = np.where(near > 0.8, d * (0.5 + rng.normal(size=n) * 1e-6) * np.sign(dy), dy)
    xj, yj = np.mod(xi + dx, L), np.mod(yi + dy, L)
    ok = (xj < L) & (yj < L) & (dx > 1e-3 * d)
    (ci, xf), (ri, yf) = in_cell(xi, a, inv_a, nc), in_cell(yi, a, inv_a, nc)
    (cj, xg), (rj, yg) = in_cell(xj, a, inv_a, nc), in_cell(yj, a, inv_a, nc)
    m = (cj - ci) % nc
    rr = rj - ri
    rr = np.where(rr > nc // 2, rr - nc, np.where(rr < -(nc // 2), rr + nc, rr))
    ok &= np.abs(rr) <= 1
    af, df, dl = f(a), f(d), f(a * 2.0 ** -20)
    ddy = (rr.astype(f) * af + (yg - yf)).astype(f)
    ay = np.abs(ddy)
    ddx = (m.astype(f) * af + (xg - xf)).astype(f)
    dele = (dl + m.astype(f) * (f(0.25) * dl)).astype(f)
    none = ay > df + dl
    doubt = (ay > df - dl) | (np.abs(ay - f(0.5 * d)) < dl) | (np.abs(ddx) < dele)
    behind = ddx < 0
    ddx = np.where(behind, ddx + f(L), ddx).astype(f)
    dele = np.where(behind, dele + f(L) * f(2.0 ** -21), dele).astype(f)
    d2 = df * df
    an, af2 = np.maximum(ay - dl, f(0)), ay + dl
    slop = df * f(2.0 ** -19) + dele
    hi = ddx - np.sqrt(np.maximum(d2 - af2 * af2 - d2 * f(2.0 ** -21), f(0))) + slop
    lo = ddx - np.sqrt(np.maximum(d2 - an * an + d2 * f(2.0 ** -21), f(0))) - slop
    kc = np.where(ay < f(0.5 * d), 0, np.where(ddy > 0, 1, 2))
    # exact, as the arrows are defined
    ey = yj - yi
    eay = np.abs(ey)
    flip = L - eay < eay
    eay = np.where(flip, L - eay, eay)
    inc = eay < d
    ekc = np.where(eay < 0.5 * d, 0, np.where((ey > 0) != flip, 1, 2))
    ex = xj - xi
    ex = np.where(ex < 0, ex + L, ex)
    tau = ex - np.sqrt(np.maximum(d * d - eay * eay, 0.0))
    assert not np.any(ok & none & inc)
    sure = ok & ~none & ~doubt
    assert np.all(inc[sure]) and np.array_equal(kc[sure], ekc[sure])
    room = 2.0 ** -21 * d
    assert np.all(lo[sure] + room < tau[sure]) and np.all(tau[sure] < hi[sure] - room)
    # and they decide nearly every pair: doubts are the ones planted at the edges
    assert np.mean((doubt & ~none)[ok & (near > 0.2) & (near < 0.8)]) < 1e-3
