"""Phase 1 with one warp per query at its edges: datasets around a sub-tile (64), a tile (512), a
super-tile (16,384) and more than one group of 32 super-tiles, k from 1 to 32, lattices full of
equal distances (more than the warp's 64-entry buffer holds), far and offset queries, and
non-finite ones, against the oracle (FP64 lists bit for bit)."""
import numpy as np
import pytest

from paper_1511_02186_gb300 import aidw, workloads
from parity import assert_parity, params_of, to_device

pytestmark = pytest.mark.gpu

SIZES = [(1, 1), (63, 32), (64, 10), (65, 32), (513, 7), (2049, 16), (16384, 32), (16385, 10),
         (540001, 10)]


@pytest.fixture(scope="module")
def ctx():
    with aidw.Context(0) as c:
        yield c


@pytest.mark.parametrize("precision", [aidw.F32C, aidw.F64])
@pytest.mark.parametrize("size", SIZES, ids=lambda s: f"n{s[0]}k{s[1]}")
def test_sizes(ctx, precision, size):
    n, k = size
    wl = workloads.small_case(n, n, 301, k=min(n, k), pattern="clustered" if n > 600 else "uniform",
                              side=100.0)
    assert_parity(ctx, wl, precision, splits=(-1, 0))


@pytest.mark.parametrize("precision", [aidw.F32C, aidw.F64])
@pytest.mark.parametrize("copies", [1, 9, 80])
@pytest.mark.parametrize("offset", [0.0, 3.0e5])
def test_equal_distances(ctx, precision, copies, offset):
    """An integer lattice, each point `copies` times (up to 80 points at one distance), queries on
    the points, between them and outside; with an offset FP32 rounding reaches the query's
    position."""
    g = np.arange(12.0)
    x, y = (np.tile(a.ravel(), copies) for a in np.meshgrid(g, g))
    rng = np.random.default_rng(copies)
    z = rng.uniform(-1, 1, x.size)
    qx = np.concatenate([g, g + 0.5, rng.uniform(-30, 40, 60)])
    qy = np.concatenate([g, g[::-1] + 0.5, rng.uniform(-30, 40, 60)])
    wl = workloads.Workload("lattice", x + offset, y + offset, z, 144.0, qx + offset, qy + offset,
                            k=10)
    assert_parity(ctx, wl, precision, splits=(-1, 0))


@pytest.mark.parametrize("precision", [aidw.F32C, aidw.F64])
def test_nonfinite_queries_give_nan_and_leave_the_others_alone(ctx, precision):
    import torch
    wl = workloads.small_case(7, 5000, 64, k=10, pattern="uniform", side=10.0)
    ds = ctx.create_dataset(wl.x, wl.y, wl.z, wl.area)
    qx, qy = to_device(wl, precision)
    p = params_of(wl, precision)
    clean = ctx.interpolate(ds, qx, qy, p, splits=(-1, 0))[0]
    bad = [3, 31, 32, 63]
    qx[bad[0]], qy[bad[1]], qx[bad[2]], qy[bad[3]] = (float("nan"), float("nan"), float("inf"),
                                                      float("-inf"))
    z = ctx.interpolate(ds, qx, qy, p, splits=(-1, 0))[0]
    keep = torch.ones(64, dtype=torch.bool, device="cuda")
    keep[bad] = False
    assert torch.isnan(z[bad]).all()
    assert torch.equal(z[keep], clean[keep])
    assert ctx.check_device_errors() == aidw.OK
    ds.destroy()
