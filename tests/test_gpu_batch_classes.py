"""Batch items whose phase 2 runs by power classes (batched.cu has its own form of them: two classes
in one region): item sizes around the least of the class route, every integer power at either end
level, items with all, none and part of their queries in the class, both phase-1 forms, powers
beyond FP32 (also in single calls), and queries on data points, against the oracle; alone, in the
mix and on replay the same bits."""
import numpy as np
import pytest

from paper_1511_02186_gb300 import aidw, workloads
from parity import TOL_F32, oracle_for, params_of, rel_err, to_device

pytestmark = pytest.mark.gpu

N = 30011
# Phase 1: 16 queries at a warp each up to 8,191 queries, the pruned scan from there on.
SIZES = [4095, 4096, 4097, 9001]


@pytest.fixture(scope="module")
def ctx():
    with aidw.Context(0) as c:
        yield c


def make(ctx, wl):
    import torch
    ds = ctx.create_dataset(wl.x, wl.y, wl.z, wl.area)
    qx, qy = to_device(wl, aidw.F32C)
    out, alpha = (torch.full((wl.m,), float("nan"), dtype=torch.float32, device="cuda")
                  for _ in range(2))
    return ds, qx, qy, params_of(wl, aidw.F32C), out, alpha


def check(ctx, wls):
    import torch
    items = [make(ctx, wl) for wl in wls]
    pb = ctx.batch_create(items)
    pb.launch()
    torch.cuda.synchronize()
    assert ctx.check_device_errors() == aidw.OK
    first = [(it[4].clone(), it[5].clone()) for it in items]
    for wl, (z, a) in zip(wls, first):
        ref, _ = oracle_for(wl, aidw.F32C)
        assert rel_err(z.cpu().numpy().astype(np.float64), ref).max() <= TOL_F32
        assert np.abs(a.cpu().numpy() - ref["alpha"]).max() <= 2e-6 * max(wl.levels)
    for it in items:
        it[4].fill_(float("nan"))
    pb.launch()
    torch.cuda.synchronize()
    for it, (z, _) in zip(items, first):
        assert torch.equal(it[4], z)
        it[4].fill_(float("nan"))
        ctx.interpolate_batch([it])
        torch.cuda.synchronize()
        assert torch.equal(it[4], z)
    pb.destroy()
    for it in items:
        it[0].destroy()


@pytest.mark.parametrize("levels", [
    (1, 2, 3, 4, 5), (0.5, 0.7, 1.5, 2.5, 1), (2.5, 1, 1, 1, 2), (1, 1, 1, 1, 3), (1, 1, 1, 1, 4),
    (1, 1.5, 2.5, 3.5, 4.5), (5, 3, 2, 1, 1.5), (3,) * 5, (1e-50, 1, 2, 3, 4),
    (1e-50, 1e-50, 1e-50, 1e-50, 2)], ids=lambda v: "-".join(str(a) for a in v))
def test_levels(ctx, levels):
    check(ctx, [workloads.small_case(51 + i, N, m, k=6, side=200.0, levels=levels,
                                     pattern="clustered" if i % 2 else "uniform")
                for i, m in enumerate(SIZES)])


@pytest.mark.parametrize("precision", [aidw.F32C, aidw.F64, aidw.F64X])
@pytest.mark.parametrize("level", [1e-50, 1e-300, 1e40, 1e300])
@pytest.mark.parametrize("m", [301, 7001])
def test_powers_beyond_fp32(ctx, precision, level, m):
    """All equal weights, or the nearest point's value (which the oracle's FP64 power also gives)."""
    wl = workloads.small_case(81, N, m, k=6, pattern="uniform", side=200.0, levels=(level,) * 5)
    ds, qx, qy, _, _, _ = make(ctx, wl)
    if precision != aidw.F32C:
        qx, qy = to_device(wl, precision)
    z = ctx.interpolate(ds, qx, qy, params_of(wl, precision))[0].cpu().numpy().astype(np.float64)
    src = wl.as_f32() if precision == aidw.F32C else wl
    d2 = ((src.qx[:200, None] - src.x[None, :]) ** 2 + (src.qy[:200, None] - src.y[None, :]) ** 2)
    want = np.full(m, src.z.mean()) if level < 1 else src.z[d2.argmin(axis=1)]
    m = len(want)
    scale = np.abs(src.z).mean() if level < 1 else np.abs(want)
    assert (np.abs(z[:m] - want) / np.maximum(np.abs(want), scale)).max() <= TOL_F32
    ds.destroy()


def test_queries_on_data_points(ctx):
    wls = [workloads.small_case(61 + i, N, m, k=10, pattern="clustered", side=50.0)
           for i, m in enumerate(SIZES)]
    for step, wl in zip((1, 3, 50, 2), wls):
        on = len(wl.qx[::step])
        wl.qx[::step], wl.qy[::step] = wl.x[:on], wl.y[:on]
    check(ctx, wls)


@pytest.mark.parametrize("z_scale", [1e12, 1e30])
def test_large_values(ctx, z_scale):
    wl = workloads.small_case(71, N, 4096, k=10, pattern="uniform", side=1.0)
    wl.z[:] *= z_scale
    check(ctx, [wl])
