"""The work that users of this library have it do, as cases that can be timed and compared.

A case is one call (or one burst of calls) through the public binding. Sizes, distributions and
parameters are those of the repository's own workloads (``workloads.py``, the tests and the
benchmark): data uniform in a square or clustered, smooth or lognormal values, the default
levels, k between 6 and 16, resident datasets of 1,024 to 1,048,576 points and calls of 256 to
1,048,576 queries, in FP32 (the main path), FP64 and FP64X, from device or host arrays, one at a
time, in prepared batches and through the serving queue.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1511_02186_gb300 import aidw, workloads

_contexts = {}


def _context(name: str = "calls") -> "aidw.Context":
    """One library context per kind of use for the whole process, as a program keeps it (the
    serving queue has one of its own)."""
    if name not in _contexts:
        _contexts[name] = aidw.Context(0)
    return _contexts[name]


PRECISION = {"f32": aidw.F32C, "f64": aidw.F64, "f64x": aidw.F64X}


def listed():
    return [
        # A small interpolation, the size of the repository's first workload: launch latency.
        dict(name="unit_1k_f32", kind="interpolate", precision="f32", data="uniform", n=1024,
             m=1024, k=10, queries="uniform", side=1.0, host=False, alpha=True, knn=False),
        # The same in double precision with the neighbour lists.
        dict(name="unit_1k_f64_knn", kind="interpolate", precision="f64", data="uniform",
             n=1024, m=1024, k=10, queries="uniform", side=1.0, host=False, alpha=True,
             knn=True),
        # A few points looked up against a resident dataset, from and to host memory.
        dict(name="lookup_257_host", kind="interpolate", precision="f32", data="uniform",
             n=300007, m=257, k=10, queries="uniform", side=1000.0, host=True, alpha=False,
             knn=False),
        # Data that is interpolated once: dataset upload, a grid of queries, dataset freed.
        dict(name="fresh_data_host", kind="fresh", precision="f32", data="clustered", n=200003,
             m=16768, k=10, queries="grid", side=100.0, host=True, alpha=False, knn=False),
        # A call of ordinary size against a large resident dataset.
        dict(name="mid_8k_1m", kind="interpolate", precision="f32", data="uniform", n=1048576,
             m=8192, k=10, queries="uniform", side=1000.0, host=False, alpha=False, knn=False),
        # A raster over clustered data with heavy-tailed values, with the powers used.
        dict(name="clustered_grid", kind="interpolate", precision="f32", data="clustered",
             n=262147, m=153984, k=15, queries="grid", side=1000.0, host=False, alpha=True,
             knn=False),
        # The paper's largest size class: as many queries as data points.
        dict(name="paper_1m", kind="interpolate", precision="f32", data="uniform", n=1048576,
             m=1048576, k=10, queries="uniform", side=1000.0, host=False, alpha=False,
             knn=False),
        # Double precision at an ordinary size, with the neighbour lists.
        dict(name="f64_8k_131k_knn", kind="interpolate", precision="f64", data="uniform",
             n=131072, m=8191, k=10, queries="uniform", side=1000.0, host=False, alpha=True,
             knn=True),
        # The double-float path at an ordinary size.
        dict(name="f64x_16k_262k", kind="interpolate", precision="f64x", data="clustered",
             n=262144, m=16384, k=10, queries="uniform", side=1000.0, host=False, alpha=False,
             knn=False),
        # Standard IDW (one power for every query).
        dict(name="idw_65k_300k", kind="idw", precision="f32", data="uniform", n=300007,
             m=65535, k=1, queries="uniform", side=1000.0, host=False, alpha=False, knn=False),
        # Many independent datasets of uneven sizes in one prepared launch.
        dict(name="batch_64", kind="batch", precision="f32", count=64, n_lo=1024, n_hi=262144,
             m_lo=1024, m_hi=65536),
        # A burst of requests of uneven sizes into the serving queue, host arrays, until the
        # last answer is back.
        dict(name="served_burst", kind="served", precision="f32", datasets=8, requests=24,
             n_lo=16384, n_hi=1048576, m_lo=256, m_hi=65536),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["interpolate"] * 5 + ["interpolate64"] * 2 + ["fresh", "idw", "batch",
                                                                      "served"])
    if kind == "batch":
        n_lo, m_lo = _log_int(rng, 1024, 8192), _log_int(rng, 1024, 4096)
        return dict(kind="batch", precision="f32", count=rng.randint(3, 64), n_lo=n_lo,
                    n_hi=_log_int(rng, 16384, 262144), m_lo=m_lo,
                    m_hi=_log_int(rng, 8192, 65536))
    if kind == "served":
        return dict(kind="served", precision="f32", datasets=rng.randint(2, 8),
                    requests=rng.randint(4, 32), n_lo=16384,
                    n_hi=_log_int(rng, 65536, 1048576), m_lo=256,
                    m_hi=_log_int(rng, 2048, 65536))
    precision = rng.choice(["f64", "f64x"]) if kind == "interpolate64" else "f32"
    cap = {"f32": 2e11, "f64": 2e9, "f64x": 4e9}[precision]
    while True:
        n, m = _log_int(rng, 1024, 1048576), _log_int(rng, 200, 1048576)
        if n * m <= cap and (kind != "fresh" or n * m <= 2e10):
            break
    queries = rng.choice(["uniform", "uniform", "grid"])
    return dict(kind={"interpolate64": "interpolate"}.get(kind, kind), precision=precision,
                data=rng.choice(["uniform", "clustered"]), n=n, m=m,
                k=1 if kind == "idw" else rng.choice([6, 8, 10, 10, 12, 15, 16]),
                queries=queries, side=float(rng.choice([1, 10, 100, 1000])),
                host=kind == "fresh" or (m < 100000 and rng.random() < 0.25),
                alpha=kind == "interpolate" and rng.random() < 0.5,
                knn=precision == "f64" and m < 50000 and rng.random() < 0.5)


# ---- inputs ------------------------------------------------------------------------------

def _data(case, rng):
    n, side = case["n"], case["side"]
    if case["data"] == "uniform":
        x, y = rng.uniform(0.0, side, n), rng.uniform(0.0, side, n)
        z = workloads.smooth_values(rng, x, y, side)
    else:
        x, y = workloads.clustered_points(rng, n, side, int(rng.integers(4, 33)), 0.005 * side,
                                          0.05 * side, 0.1)
        z = rng.lognormal(0.0, 1.0, n)
    return x, y, z


def _queries(case, rng):
    m, side = case["m"], case["side"]
    if case["queries"] == "uniform":
        return rng.uniform(0.0, side, m), rng.uniform(0.0, side, m)
    # The first m cell centres, row by row, of a grid over a window of the square.
    w = max(1, int(math.isqrt(m)))
    rows = -(-m // w)
    lo, span = rng.uniform(0.0, 0.05, 2) * side, rng.uniform(0.85, 0.95) * side
    i = np.arange(m)
    return lo[0] + (i % w + 0.5) * (span / w), lo[1] + (i // w + 0.5) * (span / rows)


def _floats(case):
    return (np.float32, "f4", torch.float32) if case["precision"] == "f32" else \
        (np.float64, "f8", torch.float64)


class State:
    """What a program holds between calls; its datasets and batch go with it."""

    def __init__(self, case):
        self.case, self.ctx, self.datasets, self.batch = case, None, [], None

    def __del__(self):
        try:
            if self.batch is not None:
                self.batch.destroy()
            for d in self.datasets:
                d.destroy()
        except Exception:  # noqa: BLE001 - at interpreter exit the context may be gone
            pass


def _spread(lo, hi, i, step):
    """The i-th of a sequence spread evenly over the logarithm of [lo, hi]: the sizes are the
    case's own, the same whatever the seed."""
    return int(round(lo * (hi / lo) ** ((0.5 + i * step) % 1.0)))


def _one_of_many(rng, n, i):
    """The i-th of many datasets: side log-uniform in [10, 1000], uniform or clustered points."""
    side = float(math.exp(rng.uniform(math.log(10.0), math.log(1000.0))))
    if i % 2:
        x, y = workloads.clustered_points(rng, n, side, int(rng.integers(4, 33)), 0.005 * side,
                                          0.05 * side, 0.1)
    else:
        x, y = rng.uniform(0.0, side, n), rng.uniform(0.0, side, n)
    z = workloads.smooth_values(rng, x, y, side)
    return (*(a.astype(np.float32) for a in (x, y, z)), side)


def _prepare_batch(st, case, seed):
    st.ctx = _context()
    rng = np.random.default_rng(seed)
    items, st.outs, st.inputs = [], [], []
    for i in range(case["count"]):
        n = _spread(case["n_lo"], case["n_hi"], i, 0.6180339887)
        m = _spread(case["m_lo"], case["m_hi"], i, 0.7548776662)
        k = (6, 10, 15)[i % 3]
        x, y, z, side = _one_of_many(rng, n, i)
        ds = st.ctx.create_dataset(x, y, z, side * side, dtype="f4")
        st.datasets.append(ds)
        qx = torch.as_tensor(rng.uniform(0.0, side, m).astype(np.float32), device="cuda")
        qy = torch.as_tensor(rng.uniform(0.0, side, m).astype(np.float32), device="cuda")
        out = torch.empty(m, dtype=torch.float32, device="cuda")
        items.append((ds, qx, qy, aidw.default_params(k=k), out, None))
        st.outs.append(out)
        st.inputs.append((x, y, z, side * side, qx, qy, k))
    st.batch = st.ctx.batch_create(items)
    return st


def _prepare_served(st, case, seed):
    st.ctx = _context("serving")
    rng = np.random.default_rng(seed)
    sets = []
    for i in range(case["datasets"]):
        x, y, z, side = _one_of_many(rng, _spread(case["n_lo"], case["n_hi"], i, 0.6180339887), i)
        sets.append((x, y, z, side * side))
        st.datasets.append(st.ctx.create_dataset(x, y, z, side * side, dtype="f4"))
    st.requests, st.inputs = [], []
    for i in range(case["requests"]):
        m = _spread(case["m_lo"], case["m_hi"], i, 0.7548776662)
        d = i % len(sets)
        side = math.sqrt(sets[d][3])
        qx = rng.uniform(0.0, side, m).astype(np.float32)
        qy = rng.uniform(0.0, side, m).astype(np.float32)
        st.requests.append((st.datasets[d], qx, qy, aidw.default_params(k=10),
                            np.empty(m, np.float32)))
        st.inputs.append((*sets[d], qx, qy, 10))
    return st


def prepare(case, seed):
    st = State(case)
    if case["kind"] == "batch":
        return _prepare_batch(st, case, seed)
    if case["kind"] == "served":
        return _prepare_served(st, case, seed)
    np_t, dt, _ = _floats(case)
    rng = np.random.default_rng(seed)
    x, y, z = (a.astype(np_t) for a in _data(case, rng))
    qx, qy = (a.astype(np_t) for a in _queries(case, rng))
    area = case["side"] ** 2
    st.ctx = _context()
    st.data, st.area, st.dt = (x, y, z), area, dt
    st.params = aidw.default_params(k=case["k"], precision=PRECISION[case["precision"]])
    if case["host"]:
        st.qx, st.qy = qx, qy
    else:
        st.qx = torch.as_tensor(qx, device="cuda")
        st.qy = torch.as_tensor(qy, device="cuda")
    if case["kind"] != "fresh":
        st.datasets.append(st.ctx.create_dataset(x, y, z, area, dtype=dt))
    st.inputs = [(x, y, z, area, st.qx, st.qy, case["k"])]
    return st


# ---- one pass ----------------------------------------------------------------------------

IDW_POWER = 2.0


def run(state):
    case, ctx = state.case, state.ctx
    kind = case["kind"]
    if kind == "batch":
        state.batch.launch()
        return state.outs
    if kind == "served":
        ids = []
        for ds, qx, qy, p, out in state.requests:
            status, rid = ctx.submit(ds, qx, qy, p, out)
            if status != aidw.OK:
                raise aidw.AidwError(status, "submit")
            ids.append(rid)
        for rid in ids:
            status = ctx.wait(rid)
            if status != aidw.OK:
                raise aidw.AidwError(status, "wait")
            ctx.release(rid)
        return [r[4] for r in state.requests]
    if kind == "idw":
        return [ctx.idw(state.datasets[0], state.qx, state.qy, IDW_POWER,
                        state.params.precision)]
    if kind == "fresh":
        ds = ctx.create_dataset(*state.data, state.area, dtype=state.dt)
        out = ctx.interpolate(ds, state.qx, state.qy, state.params)[0]
        ds.destroy()
        return [out]
    z, alpha, knn = ctx.interpolate(state.datasets[0], state.qx, state.qy, state.params,
                                    want_alpha=case["alpha"], want_knn=case["knn"])
    return [v for v in (z, alpha, knn) if v is not None]


# ---- what a pass cannot do without -------------------------------------------------------

# Per pair: two differences, the squared distance (a product and a fused multiply-add), the
# logarithm, the power (a fused multiply-add), the exponential, and the two sums (an addition and
# a fused multiply-add); an fma counts as two.
FLOPS_PER_PAIR = 12


def work(case):
    if case["kind"] == "batch":
        sizes = [(_spread(case["n_lo"], case["n_hi"], i, 0.6180339887),
                  _spread(case["m_lo"], case["m_hi"], i, 0.7548776662))
                 for i in range(case["count"])]
        return {"bytes": sum(12 * n + 12 * m for n, m in sizes),
                "flops": FLOPS_PER_PAIR * sum(n * m for n, m in sizes)}
    if case["kind"] == "served":
        n = [_spread(case["n_lo"], case["n_hi"], i, 0.6180339887)
             for i in range(case["datasets"])]
        m = [_spread(case["m_lo"], case["m_hi"], i, 0.7548776662)
             for i in range(case["requests"])]
        return {"bytes": 12 * sum(n) + 12 * sum(m),
                "flops": FLOPS_PER_PAIR * sum(n[i % len(n)] * v for i, v in enumerate(m))}
    s = 4 if case["precision"] == "f32" else 8
    per_query = 3 * s + (4 if case["alpha"] else 0) + (4 * case["k"] if case["knn"] else 0)
    return {"bytes": 3 * s * case["n"] + per_query * case["m"],
            "flops": FLOPS_PER_PAIR * case["n"] * case["m"]}


# ---- the same in 64 bits -----------------------------------------------------------------

LEVELS = (1.0, 2.0, 3.0, 4.0, 5.0)
R_MAX = 2.0


def _exact_one(x, y, z, area, qx, qy, k, power=None):
    """Z and alpha of every query in float64: Eq. 1-6 of the paper over all data points."""
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    x, y, z, qx, qy = (torch.as_tensor(a).to(dev, torch.float64) for a in (x, y, z, qx, qy))
    n, m = x.shape[0], qx.shape[0]
    r_exp = 0.5 / math.sqrt(n / area)
    out = torch.empty(m, dtype=torch.float64, device=dev)
    alpha_out = torch.empty(m, dtype=torch.float64, device=dev)
    step = max(1, (1 << 26) // n)
    levels = torch.tensor(LEVELS, dtype=torch.float64, device=dev)
    for b in range(0, m, step):
        dx = qx[b:b + step, None] - x[None, :]
        dy = qy[b:b + step, None] - y[None, :]
        d2 = dx.mul_(dx).add_(dy.mul_(dy))
        del dy
        near = d2.topk(k, dim=1, largest=False, sorted=True).values
        if power is None:
            r = near.sqrt().mean(dim=1) / r_exp
            mu = 0.5 - 0.5 * torch.cos(math.pi / R_MAX * r)
            mu = torch.where(r <= 0.0, torch.zeros_like(mu), mu)
            mu = torch.where(r >= R_MAX, torch.ones_like(mu), mu)
            t = ((mu - 0.1) * 5.0).clamp(0.0, 4.0)
            seg = t.floor().clamp(max=3.0)
            lo, hi = levels[seg.long()], levels[seg.long() + 1]
            alpha = lo + (hi - lo) * (t - seg)
        else:
            alpha = torch.full_like(near[:, 0], power)
        d1 = near[:, :1]
        # Weights relative to the nearest point's; a coincident point takes all the weight.
        w = torch.where(d1 > 0.0, (d2 / d1.clamp(min=1e-300)).log_()
                        .mul_(-0.5 * alpha[:, None]).exp_(), (d2 == 0.0).to(torch.float64))
        out[b:b + step] = (w @ z) / w.sum(dim=1)
        alpha_out[b:b + step] = alpha
    return out, alpha_out


def exact(case, seed):
    w = work(case)
    if w["flops"] > FLOPS_PER_PAIR * 1.5e10:
        return None  # tens of seconds in 64 bits
    st = prepare(case, seed)
    if case["kind"] in ("batch", "served"):
        return [_exact_one(*i)[0] for i in st.inputs]
    if case["kind"] == "idw":
        return [_exact_one(*st.inputs[0], power=IDW_POWER)[0]]
    z, alpha = _exact_one(*st.inputs[0])
    got = [z]
    if case["kind"] == "interpolate" and case["alpha"]:
        got.append(alpha)
    if case["kind"] == "interpolate" and case["knn"]:
        got.append(None)
    return got
