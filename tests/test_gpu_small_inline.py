"""Small block steps whose records travel as arguments of the launch (up to 32
staged j-records and 32 i-particles) against the same step on device-resident
records, which takes the same kernel with its records in memory: the sums are
the same operations in the same order, so every bit agrees.  Sizes on both
sides of the limits, updates in the last (ragged) tile, and an update outside
the j-range of the step, which must be stored all the same."""

import numpy as np
import pytest
import torch

from paper_0902_4463_gb300 import g6gb as g6
from paper_0902_4463_gb300 import ics

pytestmark = pytest.mark.gpu

A, B = 9, 10
EPS2 = 1e-5


def _open(cid, n, st):
    g6.g6x_open_ex(cid, n + 512, 64)
    a = np.arange(n, dtype=np.int32)
    g6.g6x_set_j_particles(cid, a, a, st["tj"], st["m"], st["j0"] / 6, st["a0"] / 2, st["v0"],
                           st["x0"])
    g6.g6x_set_j_dev(cid, 0, 0)


def _update(cid, k, st, shift):
    g6.g6x_set_j_particles(cid, k, k, np.zeros(len(k)), st["m"][k], st["j0"][k] / 6,
                           st["a0"][k] / 2, st["v0"][k], st["x0"][k] + shift)


@pytest.mark.parametrize("n", [100, 1024, 33000, 140001])
def test_records_in_the_arguments_give_the_same_bits(n):
    from paper_0902_4463_gb300 import build
    build.build()
    st = ics.taylor_state(n, 5, 0.25)
    perm = ics.permutation(n, 6)
    _open(A, n, st)
    _open(B, n, st)
    try:
        for q, (nst, ni) in enumerate([(0, 1), (1, 7), (31, 16), (32, 17), (33, 32), (5, 33),
                                       (32, 32)]):
            k = np.unique(np.append(perm[q * 40:q * 40 + nst], n - 1 if nst else [])[-nst or 1:])
            k = k.astype(np.int32)[:nst]
            act = perm[-ni:].astype(np.int32)
            t = 0.25 + q / 64.0
            rec = np.zeros(ni, dtype=g6.IREC)
            rec["x"], rec["v"], rec["index"] = st["x0"][act], st["v0"][act], act
            if nst:
                for cid in (A, B):
                    _update(cid, k, st, 1e-3 * (q + 1))
            g6.g6_set_ti(A, t)
            g6.g6calc_firsthalf(A, n, ni, act, st["x0"][act], st["v0"][act], EPS2)
            acc, jerk, pot, nnb = g6.g6calc_lasthalf2(A, n, ni, EPS2)
            d = torch.from_numpy(rec.view(np.uint8).reshape(ni, 64)).cuda()
            o = torch.zeros((ni, 64), dtype=torch.uint8, device="cuda")
            torch.cuda.synchronize()
            g6.g6x_set_j_dev(B, 0, 0)
            g6.g6x_calc_dev(B, t, n, ni, d.data_ptr(), EPS2, 0, o.data_ptr())
            g6.g6x_sync(B)
            assert g6.g6x_last_config(A) == g6.g6x_last_config(B)
            r = o.cpu().numpy().view(g6.OUT)[:, 0]
            for got, want in ((acc, r["acc"]), (jerk, r["jerk"]), (pot, r["pot"]),
                              (nnb, r["nnb"])):
                assert np.array_equal(got, want), (nst, ni)
        # an update beyond the step's j-range is stored for the next step
        far = np.array([n], dtype=np.int32)
        x = np.array([[50.0, 0, 0]])
        z = np.zeros((1, 3))
        g6.g6x_set_j_particles(A, far, far, 0.25, np.array([1.0]), z, z, z, x)
        near = n // 2
        for nj in (near, n + 1):
            act = perm[:3].astype(np.int32)
            g6.g6_set_ti(A, 0.25)
            g6.g6calc_firsthalf(A, nj, 3, act, x.repeat(3, 0) + 0.5, z.repeat(3, 0), EPS2)
            acc, jerk, pot, nnb = g6.g6calc_lasthalf2(A, nj, 3, EPS2)
            assert (nnb == n).all() == (nj == n + 1)
    finally:
        g6.g6_close(A)
        g6.g6_close(B)
