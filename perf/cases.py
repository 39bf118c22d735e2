"""The work that a user of this library has it do, as cases that can be timed.

One pass of most cases is one block step through the public calls: the
particles corrected last are sent back to j-memory, the block time is set, and
the force on the active particles is asked for (so every j-particle is
predicted anew).  `api` says by which calls:

  grape    the GRAPE-6 sequence on host arrays (g6x_set_j_particles, g6_set_ti,
           g6calc_firsthalf, g6calc_lasthalf2, neighbour lists where `lists`)
  dev      the same on records in device memory (g6x_set_j_dev, g6x_calc_dev)
  batch    one g6x_batch_calc over many clusters, uneven active sets
  hermite  a whole g6h driver run: create, advance to t_end, read the state

The DS modes evaluate pairs in FP32 (their errors are some 1e-8 to 1e-7), so
their floating results are returned as float32, as a program that goes on in
that precision takes them; the all-FP64 mode's stay float64.
"""
import ctypes
import math

import numpy as np
import torch

from paper_0902_4463_gb300 import g6gb as g6
from paper_0902_4463_gb300 import ics

PREC = {"ds": g6.G6X_PREC_DS, "ds_x64": g6.G6X_PREC_DS_X64, "fp64": g6.G6X_PREC_FP64}
T_BLK = 0.25
H2 = 1e-4                 # neighbour radius 0.01
STEPS_PER_TIME = 230.0    # block steps of a particle per unit time at eta = 0.01 (Plummer)


def _step(name, api, n, m, eps2, prec="ds", lists=False, model="plummer"):
    return dict(name=name, api=api, n=n, m=m, eps2=eps2, prec=prec, lists=lists, model=model)


def listed():
    return [
        # the smallest call: a few particles of a small cluster (host latency and launches)
        _step("step_1k_7", "grape", 1024, 7, 1e-4),
        # the mean block of a 32768-particle Hermite run
        _step("step_32k_793", "grape", 32768, 793, 1e-5),
        # a core block of a cluster with primordial binaries: few particles, many j
        _step("step_128k_24", "grape", 131072, 24, 1e-8, model="binaries"),
        # the mean block of the same run with neighbour lists read back every step
        _step("lists_128k_972", "grape", 131072, 972, 1e-8, lists=True, model="binaries"),
        # small block steps against a million particles, records on the device
        _step("step_1m_16", "dev", 1048576, 16, 1e-6),
        # an odd block against an odd number of j-particles
        _step("step_1m_251", "dev", 1000003, 251, 1e-6),
        # a large block step of the block-size sweep
        _step("step_1m_2048", "dev", 1048576, 2048, 1e-6),
        # the initial force of a 131072-particle run: all on all, through host arrays
        _step("sweep_128k", "grape", 131072, 131072, 1e-8, model="binaries"),
        # the benchmark's headline: all on all at 2^20
        _step("sweep_1m", "dev", 1048576, 1048576, 1e-6),
        # the all-FP64 path on a mean block
        _step("fp64_32k_793", "grape", 32768, 793, 1e-5, prec="fp64"),
        # 256 clusters of uneven size, uneven active sets, a fifth of them idle
        dict(name="batch_256", api="batch", ncl=256, nmin=256, nmax=16384, sizes=1),
        # a whole small integration: latency of hundreds of dependent block steps
        dict(name="hermite_1k", api="hermite", n=1024, eps2=1e-4, t_end=0.0625),
    ]


def _log(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["grape"] * 4 + ["dev"] * 5 + ["lists", "fp64", "batch", "hermite"])
    if kind == "batch":
        return dict(api="batch", ncl=_log(rng, 8, 256), nmin=256,
                    nmax=rng.choice([1024, 4096, 16384]), sizes=rng.randrange(1, 1 << 20))
    if kind == "hermite":
        n = _log(rng, 256, 4096)
        return dict(api="hermite", n=n, eps2=(4.0 / n) ** 2, t_end=0.0625)
    n = _log(rng, 256, 1 << 18 if kind in ("lists", "fp64") else 1 << 20)
    most = {"grape": 131072, "dev": n, "lists": 4096, "fp64": max(1, 2_000_000_000 // n)}[kind]
    m = _log(rng, 1, min(n, most))
    c = _step("", "dev" if kind == "dev" else "grape", n, m, (4.0 / n) ** 2,
              prec="fp64" if kind == "fp64" else rng.choice(["ds", "ds", "ds", "ds_x64"]),
              lists=kind == "lists", model=rng.choice(["plummer", "binaries"]))
    del c["name"]
    return c


# ------------------------------------------------------------------ inputs --

def _inputs(case, seed):
    """j-particles at their own last times, the block corrected last (`upd`)
    and the active block (`act`, its state predicted to T_BLK in FP64)."""
    n, m = case["n"], case["m"]
    if case["model"] == "binaries":
        mass, x, v, _ = ics.plummer_with_binaries(n, seed)
        levels = (14, 20)            # the binaries' own steps
    else:
        mass, x, v = ics.plummer(n, seed)
        levels = (4, 12)
    r = np.random.default_rng([seed, 17])
    a2 = r.standard_normal((n, 3), dtype=np.float32).astype(np.float64) * 0.3
    j6 = r.standard_normal((n, 3), dtype=np.float32).astype(np.float64) * 0.5
    tj = T_BLK - np.ldexp(1.0, -r.integers(levels[0], levels[1] + 1, size=n))
    upd = r.permutation(n)[:m].astype(np.int32)
    act = r.permutation(n)[:m].astype(np.int32)
    return dict(mass=mass, x=x, v=v, a2=a2, j6=j6, tj=tj, upd=upd, act=act)


def _predicted(d, k=slice(None)):
    h = (T_BLK - d["tj"][k])[:, None]
    x, v, a2, j6 = d["x"][k], d["v"][k], d["a2"][k], d["j6"][k]
    return x + h * (v + h * (a2 + h * j6)), v + h * (2.0 * a2 + h * 3.0 * j6)


def _batch_sizes(case):
    """Cluster sizes, active counts (spread over their logarithm, a fifth of
    the clusters idle) and softenings."""
    r = np.random.default_rng([case["sizes"], 3])
    ns = np.rint(np.exp(r.uniform(math.log(case["nmin"]), math.log(case["nmax"]),
                                  case["ncl"]))).astype(np.int32)
    ni = np.zeros_like(ns)
    for k, n in enumerate(ns):
        if r.random() >= 0.2:
            ni[k] = max(1, int(n) >> int(r.integers(0, int(math.log2(n)) + 1)))
    if not ni.any():
        ni[0] = 1
    return ns, ni, (4.0 / ns) ** 2


def _batch_inputs(case, seed):
    ns, ni, eps2 = _batch_sizes(case)
    r = np.random.default_rng([seed, 5])
    cl = []
    for k, n in enumerate(ns):
        mass, x, v = ics.plummer(int(n), seed * 1009 + k,
                                 masses=ics.salpeter_masses(int(n), seed * 1013 + k))
        cl.append(dict(mass=mass, x=x, v=v, a2=r.standard_normal((n, 3)) * 0.3,
                       j6=r.standard_normal((n, 3)) * 0.5,
                       tj=T_BLK - np.ldexp(1.0, -r.integers(4, 13, size=n))))
    return ns, ni, eps2, cl


# ------------------------------------------------------------------- state --

_stream = None


def _user_stream():
    global _stream
    if _stream is None:
        _stream = torch.cuda.Stream()
    return _stream


class State:
    """What the program keeps between calls; closes its handle when dropped."""

    def __init__(self):
        self.cid = self.batch = None

    def open(self, n, m):
        for cid in range(g6.G6_MAX_CLUSTERS):
            try:
                g6.g6x_open_ex(cid, n, m)
            except g6.G6Error as e:
                if e.code != g6.G6_EBUSY:
                    raise
                continue
            self.cid = cid
            return
        raise RuntimeError("no free cluster id")

    def __del__(self):
        if self.cid is not None:
            g6.g6_close(self.cid)
        if self.batch is not None:
            self.batch.close()


def _to_gpu(rec):
    return torch.from_numpy(rec.view(np.uint8).reshape(len(rec), rec.itemsize)).cuda()


def prepare(case, seed):
    s = State()
    s.case = case
    if case["api"] == "batch":
        ns, ni, eps2, cl = _batch_inputs(case, seed)
        s.batch = g6.G6Batch(ns)
        for k, c in enumerate(cl):
            s.batch.set_j(k, c["mass"], c["x"], c["v"], c["a2"], c["j6"], c["tj"])
            xp, vp = _predicted(c)
            s.batch.set_i(k, xp, vp)
        s.ni, s.eps2, s.t = ni, eps2, np.full(len(ns), T_BLK)
        # the program's views of its clusters' results
        s.views = [np.frombuffer((ctypes.c_char * (int(i) * g6.OUT.itemsize)).from_address(
            g6.lib().g6x_batch_results(s.batch.h, k)), dtype=g6.OUT)
            for k, i in enumerate(ni) if i > 0]
        s.batch.calc(s.t, s.eps2, s.ni)          # stores the j-particles staged above
        return s
    if case["api"] == "hermite":
        s.mass, s.x, s.v = ics.plummer(case["n"], seed)
        s.open(case["n"], case["n"])
        return s
    n, m = case["n"], case["m"]
    d = _inputs(case, seed)
    s.open(n, m)
    g6.g6x_set_precision(s.cid, PREC[case["prec"]])
    u, i = d["upd"], d["act"]
    xp, vp = _predicted(d, i)
    every = np.arange(n, dtype=np.int32)
    g6.g6x_set_j_particles(s.cid, every, every, d["tj"], d["mass"], d["j6"], d["a2"], d["v"],
                           d["x"])
    if case["api"] == "grape":
        s.upd = [np.ascontiguousarray(q) for q in (u, u, d["tj"][u], d["mass"][u], d["j6"][u],
                                                   d["a2"][u], d["v"][u], d["x"][u])]
        s.act, s.xp, s.vp = i, xp, vp
        s.h2 = None
        if case["lists"]:
            s.h2 = np.full(m, H2)
            s.nbl = np.full((m, g6.G6_MAXNB), -1, dtype=np.int32)
            s.nblen = np.zeros(m, dtype=np.int32)
            s.where = [(s.nblen.ctypes.data + 4 * k, s.nbl.ctypes.data + 4 * g6.G6_MAXNB * k)
                       for k in range(m)]
        return s
    g6.g6x_set_j_dev(s.cid, 0, 0)                # stores the j-particles staged above
    g6.g6x_sync(s.cid)
    g6.g6x_set_stream(s.cid, _user_stream().cuda_stream)
    rec = np.zeros(m, dtype=g6.JREC)
    for f, q in (("x", d["x"]), ("v", d["v"]), ("a2", d["a2"]), ("j6", d["j6"]),
                 ("mass", d["mass"]), ("tj", d["tj"])):
        rec[f] = q[u]
    rec["address"] = rec["index"] = u
    s.jrec = _to_gpu(rec)
    rec = np.zeros(m, dtype=g6.IREC)
    rec["x"], rec["v"], rec["index"] = xp, vp, i
    s.irec = _to_gpu(rec)
    s.out = torch.zeros((m, g6.OUT.itemsize), dtype=torch.uint8, device="cuda")
    return s


# --------------------------------------------------------------------- run --

def _grape(s):
    c, cid = s.case, s.cid
    n, m = c["n"], c["m"]
    g6.g6x_set_j_particles(cid, *s.upd)
    g6.g6_set_ti(cid, T_BLK)
    g6.g6calc_firsthalf(cid, n, m, s.act, s.xp, s.vp, c["eps2"], s.h2)
    acc, jerk, pot, nnb = g6.g6calc_lasthalf2(cid, n, m, c["eps2"])
    if c["prec"] != "fp64":
        acc, jerk, pot = (q.astype(np.float32) for q in (acc, jerk, pot))
    out = dict(acc=acc, jerk=jerk, pot=pot, nnb=nnb)
    if c["lists"]:
        g6.g6_read_neighbour_list(cid)
        get = g6.lib().g6_get_neighbour_list
        for k, (length, entries) in enumerate(s.where):
            get(cid, k, g6.G6_MAXNB, length, entries)
        out.update(nblen=s.nblen, nbl=s.nbl)
    return out


def _dev(s):
    c = s.case
    with torch.cuda.stream(_user_stream()):
        g6.g6x_set_j_dev(s.cid, c["m"], s.jrec.data_ptr())
        g6.g6x_calc_dev(s.cid, T_BLK, c["n"], c["m"], s.irec.data_ptr(), c["eps2"], 0,
                        s.out.data_ptr())
        force = s.out.view(torch.float64)[:, :7]
        if c["prec"] != "fp64":
            force = force.to(torch.float32)
    return dict(force=force, nnb=s.out.view(torch.int32)[:, 14],
                nnr2=s.out.view(torch.float32)[:, 15])


def _batch(s):
    s.batch.calc(s.t, s.eps2, s.ni)
    r = np.concatenate(s.views)
    return dict(force=r.view(np.float64).reshape(-1, 8)[:, :7].astype(np.float32), nnb=r["nnb"])


def _hermite(s):
    c = s.case
    sim = g6.G6HSim(s.cid, s.mass, s.x, s.v, c["eps2"], 0.01)
    try:
        sim.run(c["t_end"])
        st = sim.state()
    finally:
        sim.close()
    return {k: st[k].astype(np.float32) for k in ("x", "v", "acc", "jerk")}


def run(state):
    return {"grape": _grape, "dev": _dev, "batch": _batch,
            "hermite": _hermite}[state.case["api"]](state)


def work(case):
    """Pairs at the 60 operations of the usual count; each stored j-particle
    (84 B in the DS modes, 152 B in FP64), update, i-record and result once."""
    if case["api"] == "batch":
        ns, ni, _ = _batch_sizes(case)
        on = ni > 0
        return dict(bytes=float(84 * ns[on].sum() + 128 * ni.sum()),
                    flops=60.0 * float(np.dot(ns.astype(np.float64), ni)))
    if case["api"] == "hermite":
        n = case["n"]
        steps = n * (1.0 + STEPS_PER_TIME * case["t_end"])
        return dict(bytes=n * 19 * 8.0, flops=60.0 * steps * n)
    n, m = case["n"], case["m"]
    return dict(bytes=float(n * (152 if case["prec"] == "fp64" else 84) + m * (120 + 64 + 64)),
                flops=60.0 * n * m)


# ------------------------------------------------------------------- exact --

def _force64(xi, vi, ii, xj, vj, mj, ij, eps2):
    """Softened acceleration, jerk, potential and nearest |r|^2 in FP64."""
    dev = "cuda"
    t = [torch.as_tensor(np.ascontiguousarray(q), device=dev) for q in (xi, vi, xj, vj, mj)]
    xi, vi, xj, vj, mj = t
    ii = torch.as_tensor(np.asarray(ii, dtype=np.int64), device=dev)
    ij = torch.as_tensor(np.asarray(ij, dtype=np.int64), device=dev)
    m, n = len(xi), len(xj)
    out = torch.empty((m, 7), dtype=torch.float64, device=dev)
    nn = torch.empty(m, dtype=torch.float64, device=dev)
    rows = max(1, (1 << 24) // n)
    for k0 in range(0, m, rows):
        k = slice(k0, min(m, k0 + rows))
        dx = [xj[None, :, d] - xi[k, None, d] for d in range(3)]
        du = [vj[None, :, d] - vi[k, None, d] for d in range(3)]
        r2 = dx[0] * dx[0]
        rv = dx[0] * du[0]
        for d in (1, 2):
            r2.addcmul_(dx[d], dx[d])
            rv.addcmul_(dx[d], du[d])
        own = ij[None, :] == ii[k, None]
        r2.masked_fill_(own, math.inf)
        nn[k] = r2.min(dim=1).values
        ri = (r2 + eps2).rsqrt_()
        mr = mj[None, :] * ri
        ri.mul_(ri)
        mr3 = mr * ri
        rv.mul_(ri).mul_(-3.0)
        for d in range(3):
            out[k, d] = (mr3 * dx[d]).sum(dim=1)
            out[k, 3 + d] = du[d].addcmul_(rv, dx[d]).mul_(mr3).sum(dim=1)
        out[k, 6] = -mr.sum(dim=1)
    return out, nn


def _hermite64(m, x, v, eps2, eta, t_end, dt_max=2.0 ** -4):
    """Block-time-step 4th-order Hermite integration (Makino & Aarseth 1992
    corrector, Aarseth 1985 steps quantised to powers of two) in FP64."""
    n = len(m)
    ids = np.arange(n)

    def force(k, xk, vk, xj, vj):
        f, _ = _force64(xk, vk, ids[k], xj, vj, m, ids, eps2)
        f = f.cpu().numpy()
        return f[:, :3], f[:, 3:6]

    def size(q):
        return np.sqrt((q * q).sum(axis=1))

    x, v = x.copy(), v.copy()
    a, j = (q.copy() for q in force(ids, x, v, x, v))
    t = np.zeros(n)
    dt = np.full(n, dt_max)
    req = eta / 10.0 * size(a) / size(j)
    while (dt > req).any():
        dt[dt > req] *= 0.5
    while True:
        tb = (t + dt).min()
        if tb > t_end:
            return x, v, a, j
        k = np.nonzero(t + dt == tb)[0]
        h = (tb - t)[:, None]
        xp = x + h * (v + h * (a / 2.0 + h * (j / 6.0)))
        vp = v + h * (a + h * (j / 2.0))
        a1, j1 = force(k, xp[k], vp[k], xp, vp)
        h = h[k]
        da = a[k] - a1
        d2 = (-6.0 * da - h * (4.0 * j[k] + 2.0 * j1)) / h ** 2
        d3 = (12.0 * da + 6.0 * h * (j[k] + j1)) / h ** 3
        x[k] = xp[k] + h ** 4 * (d2 / 24.0 + h * d3 / 120.0)
        v[k] = vp[k] + h ** 3 * (d2 / 6.0 + h * d3 / 24.0)
        a[k], j[k], t[k] = a1, j1, tb
        d2 = d2 + h * d3
        req = np.sqrt(eta * (size(a1) * size(d2) + size(j1) ** 2)
                      / (size(j1) * size(d3) + size(d2) ** 2))
        new = dt[k]
        up = (req >= 2.0 * new) & (2.0 * new <= dt_max) & (np.floor(tb / (2.0 * new))
                                                           == tb / (2.0 * new))
        new[up] *= 2.0
        while (new > req).any():
            new[new > req] *= 0.5
        dt[k] = new


def exact(case, seed):
    if case["api"] == "hermite":
        m, x, v = ics.plummer(case["n"], seed)
        return dict(zip(("x", "v", "acc", "jerk"),
                        _hermite64(m, x, v, case["eps2"], 0.01, case["t_end"])))
    if case["api"] == "batch":
        ns, ni, eps2, cl = _batch_inputs(case, seed)
        f = []
        for k, c in enumerate(cl):
            if ni[k] > 0:
                x, v = _predicted(c)
                ids = np.arange(ns[k])
                f.append(_force64(x[:ni[k]], v[:ni[k]], ids[:ni[k]], x, v, c["mass"], ids,
                                  eps2[k])[0].cpu())
        return dict(force=torch.cat(f), nnb=None)
    if float(case["n"]) * case["m"] > 3e10:
        return None
    d = _inputs(case, seed)
    x, v = _predicted(d)
    i = d["act"]
    f, nn = _force64(x[i], v[i], i, x, v, d["mass"], np.arange(case["n"]), case["eps2"])
    if case["api"] == "dev":
        return dict(force=f, nnb=None, nnr2=nn)
    f = f.cpu().numpy()
    out = dict(acc=f[:, :3], jerk=f[:, 3:6], pot=f[:, 6], nnb=None)
    if case["lists"]:
        out.update(nblen=None, nbl=None)
    return out
