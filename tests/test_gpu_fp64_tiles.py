"""The all-FP64 force (K2d) at the edges of its i-tiles (8, 16, 32) and of its
sub-tiles of 64 j-particles, against the FP64 oracle, and the arguments its
reciprocal square root hands to the library's (zero, subnormal).

Tolerances: FP64 rounding over N terms, median 1e-12 and max 1e-10 relative,
as for every FP64 force."""
import numpy as np
import pytest

from paper_0902_4463_gb300 import g6gb as g6
from paper_0902_4463_gb300 import ics
from tests.gpu_helpers import load_j, rel_err_vec, sweep

pytestmark = pytest.mark.gpu

CID = 8


def _open(n, m):
    from paper_0902_4463_gb300 import build
    build.build()
    g6.g6x_open_ex(CID, n, m)
    g6.g6x_set_precision(CID, g6.G6X_PREC_FP64)


@pytest.mark.parametrize("n", [2, 63, 64, 65, 257, 3001])
def test_tile_edges_against_the_oracle(orc, n):
    st = ics.taylor_state(n, n, 0.5)
    idx = np.arange(n, dtype=np.int32)
    _open(n, n)
    try:
        load_j(CID, st["x0"], st["v0"], st["m"], st["a0"], st["j0"], st["tj"])
        xp, vp = orc.predict(st["x0"], st["v0"], st["a0"], st["j0"], st["tj"], 0.5)
        perm = ics.permutation(n, 3)
        for m in sorted({1, 7, 8, 9, 16, 17, 31, 32, 33, 40, 257, 300} & set(range(1, n + 1))):
            act = perm[:m]
            for grid in (0, 1, 7):
                g6.g6x_set_variant(CID, -1, grid)
                acc, jerk, pot, nnb = sweep(CID, n, xp[act], vp[act], act, 1e-5, 0.5)
                oa, oj, op, onn, _ = orc.force(xp[act], vp[act], act, xp, vp, st["m"], idx, 1e-5)
                for e in (rel_err_vec(acc, oa), rel_err_vec(jerk, oj),
                          np.abs(pot - op) / np.abs(op)):
                    assert np.median(e) <= 1e-12 and e.max() <= 1e-10, (m, grid, e.max())
                assert np.array_equal(nnb, onn), (m, grid)
    finally:
        g6.g6x_set_variant(CID, -1, 0)
        g6.g6_close(CID)


@pytest.mark.parametrize("sep", [0.0, 1e-160, 1e-150, 1e-3, 1e150])
def test_pair_without_softening_at_extreme_separations(sep):
    # two bodies on the x axis, masses 1: pot = -1/sep, |a| = 1/sep^2 as far
    # as FP64 holds them; coincident bodies give an infinite potential and an
    # undefined acceleration
    x = np.array([[0.0, 0, 0], [sep, 0, 0]])
    z = np.zeros((2, 3))
    _open(2, 2)
    try:
        load_j(CID, x, z, np.ones(2))
        acc, jerk, pot, nnb = sweep(CID, 2, x, z, np.arange(2), 0.0, 0.0)
    finally:
        g6.g6_close(CID)
    # (a neighbour beyond 1e15 counts as an empty slot, which is parked there)
    assert list(nnb) == ([1, 0] if sep < 1e15 else [-1, -1])
    with np.errstate(all="ignore"):
        r2 = np.float64(sep) * np.float64(sep)
        ri = 1.0 / np.sqrt(r2)                        # what FP64 keeps of 1/|r|
        a = np.float64(1.0) * ri * (ri * ri) * sep
    assert np.allclose(pot, -ri, rtol=1e-14, atol=0) if np.isfinite(ri) else np.all(pot == -ri)
    if np.isfinite(a):
        assert np.allclose(acc[:, 0], [a, -a], rtol=1e-13, atol=0)
    else:
        assert not np.isfinite(acc[:, 0]).any()
