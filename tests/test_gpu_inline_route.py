"""Which block steps carry their records in the launch's arguments (up to 32
staged j-records, all in the j-tiles of the launch, and up to 32 i-particles)
and which take them from memory: read off the names of the kernels that a
profiler saw, with the 16- and 32-wide small-block shapes pinned so that every
size reaches the choice.  Both routes give the same bits."""
import numpy as np
import pytest
import torch

from paper_0902_4463_gb300 import g6gb as g6
from paper_0902_4463_gb300 import ics

pytestmark = pytest.mark.gpu

A, B = 9, 10
EPS2 = 1e-5
N = 3000                                      # 12 j-tiles


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_0902_4463_gb300 import build
    build.build()


def _open(cid, n, st):
    g6.g6x_open_ex(cid, n, 64)
    a = np.arange(n, dtype=np.int32)
    g6.g6x_set_j_particles(cid, a, a, st["tj"], st["m"], st["j0"] / 6, st["a0"] / 2, st["v0"],
                           st["x0"])
    g6.g6x_set_j_dev(cid, 0, 0)
    g6.g6x_sync(cid)


def _kernels(step):
    """(result of step(), names of the kernels it launched); step leaves the
    same state each time, so a trace that came back empty is taken again"""
    from torch.profiler import ProfilerActivity, profile
    for _ in range(5):
        torch.zeros(1, device="cuda")
        torch.cuda.synchronize()
        with profile(activities=[ProfilerActivity.CUDA, ProfilerActivity.CPU]) as p:
            r = step()
            torch.cuda.synchronize()
        names = [e.name for e in p.events() if "k_force" in e.name or "k_predict" in e.name]
        if any("k_force" in k for k in names):
            return r, names
    pytest.skip("no kernel records from the profiler")


def _step(cid, st, nj, upd, act, t, shift):
    if len(upd):
        g6.g6x_set_j_particles(cid, upd, upd, np.zeros(len(upd)), st["m"][upd],
                               st["j0"][upd] / 6, st["a0"][upd] / 2, st["v0"][upd],
                               st["x0"][upd] + shift)
    g6.g6_set_ti(cid, t)
    g6.g6calc_firsthalf(cid, nj, len(act), act, st["x0"][act], st["v0"][act], EPS2)
    return g6.g6calc_lasthalf2(cid, nj, len(act), EPS2)


def _step_dev(cid, st, nj, upd, act, t, shift):
    """The same on i-records in device memory: never in the arguments."""
    if len(upd):
        g6.g6x_set_j_particles(cid, upd, upd, np.zeros(len(upd)), st["m"][upd],
                               st["j0"][upd] / 6, st["a0"][upd] / 2, st["v0"][upd],
                               st["x0"][upd] + shift)
    rec = np.zeros(len(act), dtype=g6.IREC)
    rec["x"], rec["v"], rec["index"] = st["x0"][act], st["v0"][act], act
    d = torch.from_numpy(rec.view(np.uint8).reshape(len(act), 64)).cuda()
    o = torch.zeros((len(act), 64), dtype=torch.uint8, device="cuda")
    torch.cuda.synchronize()
    g6.g6x_calc_dev(cid, t, nj, len(act), d.data_ptr(), EPS2, 0, o.data_ptr())
    g6.g6x_sync(cid)
    r = o.cpu().numpy().view(g6.OUT)[:, 0]
    return r["acc"], r["jerk"], r["pot"], r["nnb"]


# (staged, active, j-range, update far from the others, in the arguments)
CASES = [(0, 1, N, None, True), (1, 7, N, None, True), (31, 16, N, None, True),
         (32, 16, N, None, True), (33, 16, N, None, False), (32, 17, N, None, True),
         (32, 31, N, None, True), (0, 32, N, None, True), (33, 32, N, None, False),
         (5, 33, N, None, False),
         (4, 8, 700, 767, True),               # the last tile of the range, beyond its end
         (4, 8, 700, 768, False),              # the first tile that the launch does not read
         (4, 8, 700, N - 1, False)]


@pytest.mark.parametrize("staged,active,nj,far,inline", CASES)
def test_the_route_and_its_bits(staged, active, nj, far, inline):
    st = ics.taylor_state(N, 5, 0.25)
    _open(A, N, st)
    _open(B, N, st)
    try:
        upd = np.arange(staged, dtype=np.int32) * 17
        if far is not None:
            upd[-1] = far
        act = (np.arange(active, dtype=np.int32) * 13 + 5) % min(nj, 650)
        shape = 37 if active <= 8 else 28 if active <= 16 else 29 if active <= 32 else 30
        assert g6.g6x_variant_info(shape)["ws"] == 1
        for cid in (A, B):
            g6.g6x_set_variant(cid, shape, 0)
        got, names = _kernels(lambda: _step(A, st, nj, upd, act, 0.25, 1e-3))
        force = [k for k in names if "k_force_ws" in k]
        assert len(force) == 1
        assert ("WsInline" in force[0]) == inline, force
        assert ("k_predict" in " ".join(names)) == (far is not None and not inline), names
        want = _step_dev(B, st, nj, upd, act, 0.25, 1e-3)
        # a step over all particles sees every update, wherever it was stored
        t = 0.25 + 1 / 64
        none = np.zeros(0, dtype=np.int32)
        got = got + _step(A, st, N, none, act, t, 0.0)
        want = want + _step_dev(B, st, N, none, act, t, 0.0)
        for q, (g, w) in enumerate(zip(got, want)):
            assert np.array_equal(g, w), q
        assert g6.g6x_last_config(A) == g6.g6x_last_config(B)
    finally:
        for cid in (A, B):
            g6.g6x_set_variant(cid, -1, 0)
            g6.g6_close(cid)


def test_device_records_never_travel_in_the_arguments():
    st = ics.taylor_state(N, 5, 0.25)
    _open(B, N, st)
    try:
        act = np.arange(7, dtype=np.int32)
        _, names = _kernels(lambda: _step_dev(B, st, N, act, act, 0.25, 1e-3))
        force = [k for k in names if "k_force_ws" in k]
        assert len(force) == 1 and "WsNone" in force[0], names
    finally:
        g6.g6_close(B)
