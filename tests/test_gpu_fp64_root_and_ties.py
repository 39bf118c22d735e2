"""The all-FP64 force kernel's reciprocal square root against exact integer
arithmetic, its nearest neighbour where distances are equal or not a number,
and ties in the shapes with neighbour lists.

One j-particle of mass 1 at the origin and no softening: the potential of an
i-particle at (d, 0, 0) is -1 / sqrt(fl(d d)) and nothing else, so one call
gives the reciprocal root of as many arguments as there are i-particles.

Bound for the root y = y0 + y0 e (1/2 + 3/8 e), e = 1 - s y0^2, in units in
the last place: the iteration leaves 5/16 e^3, below 2^-60 of the result for an
approximation good to 2^-20; the last fused multiply-add rounds once (1/2
unit); the rounding of s y0 (2^-53 relative) reaches the result halved, as
2^-54 of it, which is at most 1/2 unit (just below a power of two); the small
terms round by 2^-20 of that.  Together below 1.001; the test allows 1.01.  The library's
function, which takes zero, subnormal and infinite arguments, is documented to
1 unit; 2 are allowed."""
import math

import numpy as np
import pytest

from paper_0902_4463_gb300 import g6gb as g6

pytestmark = pytest.mark.gpu

CID = 8
INF = float("inf")


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_0902_4463_gb300 import build
    build.build()


def _roots(d, variant):
    """-potential at (d, 0, 0) of a unit mass at the origin."""
    n = len(d)
    x = np.zeros((n, 3))
    x[:, 0] = d
    z = np.zeros((n, 3))
    g6.g6x_open_ex(CID, 1, n)
    try:
        g6.g6x_set_precision(CID, g6.G6X_PREC_FP64)
        g6.g6x_set_variant(CID, variant, 0)
        g6.g6x_set_j_particles(CID, np.zeros(1, dtype=np.int32), np.zeros(1, dtype=np.int32), 0.0,
                               np.ones(1), z[:1], z[:1], z[:1], z[:1])
        g6.g6_set_ti(CID, 0.0)
        g6.g6calc_firsthalf(CID, 1, n, np.arange(1, n + 1, dtype=np.int32), x, z, 0.0)
        pot = g6.g6calc_lasthalf2(CID, 1, n, 0.0)[2]
        assert g6.g6x_last_config(CID)["variant"] == variant
        return -pot
    finally:
        g6.g6x_set_variant(CID, -1, 0)
        g6.g6_close(CID)


def _ulps(y, s):
    """|y - 1/sqrt(s)| in units in the last place of y, by integers."""
    ny, ey = math.frexp(y)
    ny, ey = int(ny * 2 ** 53), ey - 53                # y = ny 2^ey, 2^52 <= ny < 2^53
    ms, es = math.frexp(s)
    ms, es = int(ms * 2 ** 53), es - 53
    if es % 2:
        ms, es = ms * 2, es - 1                        # s = ms 2^es, es even
    # 1/sqrt(s) = 2^(-es/2) / sqrt(ms); r = floor(2^k / sqrt(ms))
    k = 180
    r = math.isqrt((1 << (2 * k)) // ms)
    got = ny << 60
    want_shift = -es // 2 - k - ey + 60                # want = r 2^(-es/2 - k), in 2^(ey - 60)
    want = r << want_shift if want_shift >= 0 else r >> -want_shift
    return abs(got - want) / 2.0 ** 60


def test_the_measure_of_error():
    # a correctly rounded value is within half a unit, a neighbour beyond it
    for s in (2.0, 3.0, 0.7, 1e-300, 1e300, 2.0 ** -1022):
        y = 1.0 / math.sqrt(s)
        assert _ulps(y, s) <= 1.5
        assert _ulps(np.nextafter(np.nextafter(np.nextafter(y, INF), INF), INF), s) >= 1.5
    assert _ulps(0.5, 4.0) == 0.0


@pytest.mark.parametrize("variant", [7, 38, 39])
def test_reciprocal_root_over_mantissas_and_exponents(variant):
    r = np.random.default_rng(64 + variant)
    # separations whose squares cover [1, 4) finely, then every binary
    # exponent of a normal square
    m = np.concatenate([np.linspace(1.0, 2.0, 20001), r.uniform(1.0, 2.0, 20000),
                        1.0 + np.arange(64) * 2.0 ** -52, 2.0 - (1 + np.arange(64)) * 2.0 ** -52])
    e = np.concatenate([np.zeros(len(m), dtype=int), np.repeat(np.arange(-511, 512), 12)])
    m = np.concatenate([m, r.uniform(1.0, 2.0, 12 * 1023)])
    d = np.ldexp(m, e)
    s = d * d
    ok = (s >= 2.0 ** -1022) & (s < INF)
    d, s = d[ok], s[ok]
    assert s.min() < 2.0 ** -1020 and s.max() > 2.0 ** 1022
    worst = max(_ulps(float(y), float(q)) for y, q in zip(_roots(d, variant), s))
    print("worst error %.3f ulp over %d arguments" % (worst, len(s)))
    assert worst <= 1.01


@pytest.mark.parametrize("variant", [7, 38, 39])
def test_reciprocal_root_where_the_library_takes_over(variant):
    # squares on both sides of the smallest normal number, and of infinity
    lo = [2.0 ** -511, np.nextafter(2.0 ** -511, 0), 2.0 ** -512, 1.3 * 2.0 ** -530, 2.0 ** -537,
          np.nextafter(2.0 ** -511, 1)]
    hi = [np.sqrt(np.finfo(float).max), 1.3e154]
    d = np.array(lo + hi + [0.0, 1e-200, 1e155, INF])
    with np.errstate(over="ignore", under="ignore"):
        s = d * d
    y = _roots(d, variant)
    for q, (yy, ss) in enumerate(zip(y, s)):
        if ss == 0.0:
            assert yy == INF, (q, yy)
        elif ss == INF:
            assert yy == 0.0, (q, yy)
        else:
            assert _ulps(float(yy), float(ss)) <= (1.01 if ss >= 2.0 ** -1022 else 2.0), (q, yy)


def _points(n, seed):
    r = np.random.default_rng(seed)
    x = r.integers(0, 8, size=(n, 3)).astype(np.float64)
    return x, r.permutation(4 * n)[:n].astype(np.int32), r.permutation(n)


def _expected(x, index, act):
    xi = x.astype(np.int64)
    out = np.empty(len(act), dtype=np.int32)
    for q, k in enumerate(act):
        d = ((xi - xi[k]) ** 2).sum(axis=1)
        d[index == index[k]] = 1 << 30
        j = int(np.argmin(d))                           # the first of equal ones
        out[q] = index[j] if d[j] < 1 << 30 else -1
    return out


@pytest.mark.parametrize("n", [1, 2, 33, 63, 65, 257, 1300])
def test_ties_in_fp64_and_in_list_shapes(n):
    x, index, perm = _points(n, n)
    z = np.zeros((n, 3))
    g6.g6x_open_ex(CID, n, n)
    try:
        g6.g6x_set_j_particles(CID, np.arange(n), index, 0.0, np.full(n, 1.0 / n), z, z, z, x)
        want = _expected(x, index, perm)
        seen = 0
        for v in range(g6.g6x_variant_count()):
            info = g6.g6x_variant_info(v)
            if info["prec"] != g6.G6X_PREC_FP64 and not info["list"]:
                continue
            g6.g6x_set_precision(CID, info["prec"])
            for grid in (0, 1, 5):
                g6.g6x_set_variant(CID, v, grid)
                g6.g6_set_ti(CID, 0.0)
                # a radius of 0.5: the coincident particles (at distance 0)
                g6.g6calc_firsthalf(CID, n, n, index[perm], x[perm], z[perm], 2.0 ** -10,
                                    np.full(n, 0.25) if info["list"] else None)
                nnb = g6.g6calc_lasthalf2(CID, n, n, 2.0 ** -10)[3]
                assert g6.g6x_last_config(CID)["variant"] == v
                assert np.array_equal(nnb, want), (v, grid, info)
                seen += 1
        assert seen >= 3 * (4 + 7)
    finally:
        g6.g6x_set_variant(CID, -1, 0)
        g6.g6_close(CID)


@pytest.mark.parametrize("variant", [7, 38, 39, 8])
@pytest.mark.parametrize("nan", [float("nan"), -float("nan")])
def test_a_nan_distance_is_never_the_nearest(variant, nan):
    # Velocities and accelerations of 0, so only the positions that are not a
    # number (either sign) make distances that are not; the NaN particles come
    # first, between and last, one per j-group's share at least
    n = 140
    x = np.zeros((n, 3))
    x[:, 0] = np.arange(n)
    bad = np.arange(n) % 3 != 1
    x[bad, 1] = nan
    index = np.arange(n, dtype=np.int32) * 2 + 1
    z = np.zeros((n, 3))
    act = np.array([1, 4, 64, 139], dtype=np.int32)
    act = act[~bad[act]]
    g6.g6x_open_ex(CID, n, n)
    try:
        g6.g6x_set_precision(CID, g6.G6X_PREC_FP64)
        g6.g6x_set_variant(CID, variant, 0)
        g6.g6x_set_j_particles(CID, np.arange(n, dtype=np.int32), index, 0.0, np.ones(n), z, z, z,
                               x)
        g6.g6_set_ti(CID, 0.0)
        g6.g6calc_firsthalf(CID, n, len(act), index[act], x[act], z[act], 0.0,
                            np.full(len(act), 10.0) if variant == 8 else None)
        nnb = g6.g6calc_lasthalf2(CID, n, len(act), 0.0)[3]
    finally:
        g6.g6x_set_variant(CID, -1, 0)
        g6.g6_close(CID)
    good = np.nonzero(~bad)[0]
    for k, got in zip(act, nnb):
        d = np.abs(good - k).astype(float)
        d[good == k] = INF
        assert got == index[good[np.argmin(d)]], (k, got)
