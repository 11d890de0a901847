"""FP32 phase 2 by power classes where d^-power times a value leaves FP32's range: small values at
large distances, and coordinates far from 0 beside small distances, in single calls and batches,
against the oracle."""
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
    import torch
    ref, _ = oracle_for(wl, aidw.F32C)
    ds = ctx.create_dataset(wl.x, wl.y, wl.z, wl.area)
    qx, qy = to_device(wl, aidw.F32C)
    single = ctx.interpolate(ds, qx, qy, params_of(wl, aidw.F32C))[0]
    out = torch.full_like(single, float("nan"))
    ctx.interpolate_batch([(ds, qx, qy, params_of(wl, aidw.F32C), out, None)])
    assert ctx.check_device_errors() == aidw.OK
    ds.destroy()
    for z in (single, out):
        assert rel_err(z.cpu().numpy().astype(np.float64), ref).max() <= TOL_F32


@pytest.mark.parametrize("levels", [(1, 2, 3, 4, 5), (1,) * 5, (2,) * 5, (3,) * 5, (4,) * 5,
                                    (5,) * 5], ids=lambda v: "-".join(str(a) for a in v))
@pytest.mark.parametrize("side", [1e3, 1e5, 1e6, 1e7])
@pytest.mark.parametrize("z_scale", [1e-20, 1e-30])
def test_small_values(ctx, levels, side, z_scale):
    wl = workloads.small_case(41, N, M, k=10, pattern="uniform", side=side, levels=levels)
    wl.z[:] = (1.5 + np.sin(np.arange(N))) * z_scale
    check(ctx, wl)


@pytest.mark.parametrize("levels", [(1,) * 5, (5, 4, 3, 2, 1)])
@pytest.mark.parametrize("span", [1e-8, 1e-3, 1e3])
def test_points_on_a_line_far_from_the_origin(ctx, levels, span):
    """All x are 2^65 and the distances lie in y: the scaled x would overflow."""
    wl = workloads.small_case(42, N, M, k=10, pattern="uniform", side=1.0, levels=levels)
    wl.x[:] = wl.qx[:] = 2.0 ** 65
    wl.y[:] *= span
    wl.qy[:] *= span
    check(ctx, wl)


@pytest.mark.parametrize("side", [10.0, 1e3, 1e5])
@pytest.mark.parametrize("values", ["zeros", "tiny", "huge", "wide", "mostly zero"])
def test_value_ranges(ctx, side, values):
    """The FP32 copy holds the values times a power of two: none at all, the ends of FP32's range,
    values over 30 orders of magnitude in one dataset, and nearly all 0."""
    wl = workloads.small_case(43, N, M, k=10, pattern="uniform", side=side)
    rng = np.random.default_rng(5)
    wl.z[:] = {"zeros": np.zeros(N), "tiny": rng.uniform(1, 2, N) * 2e-37,
               "huge": rng.uniform(-1, 1, N) * 1e33, "wide": 10.0 ** rng.uniform(-30, 0, N),
               "mostly zero": (rng.uniform(0, 1, N) < 1e-3) * rng.uniform(1, 2, N)}[values]
    if values == "zeros":
        ds = ctx.create_dataset(wl.x, wl.y, wl.z, wl.area)
        qx, qy = to_device(wl, aidw.F32C)
        assert (ctx.interpolate(ds, qx, qy, params_of(wl, aidw.F32C))[0] == 0.0).all()
        ds.destroy()
    else:
        check(ctx, wl)
