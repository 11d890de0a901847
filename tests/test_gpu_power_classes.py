"""FP32 phase 2 by power classes: calls large enough for it, with integer and other end levels,
queries on data points, values too large for the unscaled sums and coordinates whose powers
leave their range, against the oracle; each power's loop with queries of every class in one
call."""
import numpy as np
import pytest

from paper_1511_02186_gb300 import aidw, workloads
from parity import TOL_F32, oracle_for, params_of, rel_err, to_device

pytestmark = pytest.mark.gpu

N, M = 50021, 4099  # just above the class route's least size


@pytest.fixture(scope="module")
def ctx():
    with aidw.Context(0) as c:
        yield c


def check(ctx, wl):
    ref, _ = oracle_for(wl, aidw.F32C)
    ds = ctx.create_dataset(wl.x, wl.y, wl.z, wl.area)
    qx, qy = to_device(wl, aidw.F32C)
    z = ctx.interpolate(ds, qx, qy, params_of(wl, aidw.F32C))[0].cpu().numpy().astype(np.float64)
    assert ctx.check_device_errors() == aidw.OK
    ds.destroy()
    assert rel_err(z, ref).max() <= TOL_F32


@pytest.mark.parametrize("levels", [(1, 2, 3, 4, 5), (2, 2, 2, 2, 2), (3, 2, 1, 2, 4),
                                    (5, 4, 3, 2, 1), (4, 1, 1, 1, 3), (1, 1, 1, 1, 6),
                                    (0.5, 1, 2, 3, 2.5), (1, 7, 0.3, 2, 5)],
                         ids=lambda v: "-".join(str(a) for a in v))
@pytest.mark.parametrize("pattern", ["uniform", "clustered"])
def test_levels(ctx, levels, pattern):
    check(ctx, workloads.small_case(31, N, M, k=6, pattern=pattern, side=200.0, levels=levels))


@pytest.mark.parametrize("power", [1.0, 2.0, 3.0, 4.0, 5.0])
def test_constant_power(ctx, power):
    wl = workloads.small_case(32, N, M, k=1, pattern="uniform", side=3.0, levels=(power,) * 5)
    ref, _ = oracle_for(wl, aidw.F32C)
    ds = ctx.create_dataset(wl.x, wl.y, wl.z, wl.area)
    qx, qy = to_device(wl, aidw.F32C)
    z = ctx.idw(ds, qx, qy, power).cpu().numpy().astype(np.float64)
    ds.destroy()
    assert rel_err(z, ref).max() <= TOL_F32


def test_queries_on_data_points(ctx):
    wl = workloads.small_case(33, N, M, k=10, pattern="clustered", side=50.0)
    wl.qx[::3], wl.qy[::3] = wl.x[: len(wl.qx[::3])], wl.y[: len(wl.qy[::3])]
    check(ctx, wl)


@pytest.mark.parametrize("z_scale", [1e12, 1e30])
def test_large_values(ctx, z_scale):
    wl = workloads.small_case(34, N, M, k=10, pattern="uniform", side=1.0)
    wl.z[:] = wl.z * z_scale
    check(ctx, wl)


@pytest.mark.parametrize("side", [1e-9, 1e-4, 1e9])
def test_scales(ctx, side):
    """At 1e-9 every unscaled power is out of range, at 1e-4 those of some queries are."""
    check(ctx, workloads.small_case(35, N, M, k=10, pattern="uniform", side=side))


def test_a_query_keeps_its_result_whatever_class_its_neighbours_are_in(ctx):
    """The same queries in another order give the same bits."""
    import torch
    wl = workloads.small_case(36, N, M, k=6, pattern="clustered", side=100.0)
    ds = ctx.create_dataset(wl.x, wl.y, wl.z, wl.area)
    qx, qy = to_device(wl, aidw.F32C)
    p = params_of(wl, aidw.F32C)
    z = ctx.interpolate(ds, qx, qy, p)[0]
    perm = torch.randperm(wl.m, device="cuda")
    z2 = ctx.interpolate(ds, qx[perm].contiguous(), qy[perm].contiguous(), p)[0]
    assert torch.equal(z[perm], z2)
    ds.destroy()
