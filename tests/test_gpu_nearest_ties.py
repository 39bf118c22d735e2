"""Nearest neighbours where many distances are equal (Sect. 2.5: ties go to
the lower j-slot), with particle indices that are not the slots, for every
force shape.  Coordinates are small integers and eps2 a power of two, so every
squared distance is exact in FP32 and the expected neighbour follows from
integer arithmetic alone: no tolerance."""
import numpy as np
import pytest

from paper_0902_4463_gb300 import g6gb as g6

pytestmark = pytest.mark.gpu

CID = 7
EPS2 = 2.0 ** -10


def _points(n, seed):
    r = np.random.default_rng(seed)
    x = r.integers(0, 8, size=(n, 3)).astype(np.float64)
    index = r.permutation(4 * n)[:n].astype(np.int32)     # sparse, not the slot
    return x, index, r.permutation(n)


def _expected(x, index, act):
    xi = x.astype(np.int64)
    out = np.empty(len(act), dtype=np.int32)
    for q, k in enumerate(act):
        d = ((xi - xi[k]) ** 2).sum(axis=1)
        d[index == index[k]] = 1 << 30
        j = int(np.argmin(d))                             # the first of equal ones
        out[q] = index[j] if d[j] < 1 << 30 else -1
    return out


@pytest.mark.parametrize("n", [1, 2, 33, 255, 257, 1300])
def test_ties_go_to_the_lower_slot_in_every_shape(n):
    from paper_0902_4463_gb300 import build
    build.build()
    x, index, perm = _points(n, n)
    z = np.zeros((n, 3))
    g6.g6x_open_ex(CID, n, n)
    try:
        g6.g6x_set_j_particles(CID, np.arange(n), index, 0.0, np.full(n, 1.0 / n), z, z, z, x)
        for v in range(g6.g6x_variant_count()):
            info = g6.g6x_variant_info(v)
            if info["prec"] == g6.G6X_PREC_FP64 or info["list"]:
                continue
            m = min(n, info["ti"] * info["ni_per"]) if info["ws"] else n
            act = perm[:m]
            g6.g6x_set_precision(CID, info["prec"])
            g6.g6x_set_variant(CID, v, 0)
            g6.g6_set_ti(CID, 0.0)
            g6.g6calc_firsthalf(CID, n, m, index[act], x[act], z[act], EPS2)
            nnb = g6.g6calc_lasthalf2(CID, n, m, EPS2)[3]
            assert g6.g6x_last_config(CID)["variant"] == v
            assert np.array_equal(nnb, _expected(x, index, act)), (v, info)
    finally:
        g6.g6x_set_variant(CID, -1, 0)
        g6.g6_close(CID)


@pytest.mark.parametrize("variant", range(8))
def test_ties_go_to_the_lower_slot_in_batches(variant):
    from paper_0902_4463_gb300 import build
    build.build()
    sizes = [1, 33, 257, 1300]
    b = g6.G6Batch(sizes, variant=variant)
    try:
        cl = [_points(n, n + 7) for n in sizes]
        for k, (x, _, _) in enumerate(cl):
            z = np.zeros_like(x)
            b.set_j(k, np.full(len(x), 1.0 / len(x)), x, z)
            b.set_i(k, x, z)
        b.calc(np.zeros(4), np.full(4, EPS2), np.array(sizes))
        for k, (x, _, _) in enumerate(cl):
            n = len(x)
            want = _expected(x, np.arange(n, dtype=np.int32), np.arange(n))
            assert np.array_equal(b.results(k, n)["nnb"], want), (variant, n)
    finally:
        b.close()
