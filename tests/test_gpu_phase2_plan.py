"""Phase 2 at the edges of its plan: data splits at any multiple of 32 points, point groups inside a
CTA (few queries), partly filled tiles and chunks, and the merge of many splits, against the
oracle in every precision."""
import numpy as np
import pytest

from paper_1511_02186_gb300 import aidw, workloads
from parity import TOL_F32, TOL_F64, oracle_for, params_of, rel_err, to_device

pytestmark = pytest.mark.gpu

# n: one point, around a chunk (32), a point-group step (128), a tile (256, 512), the padding
# granule (2,048); m: around a warp, a CTA with and without point groups in FP32 (64, 256, the
# switch at 2,048) and FP64 (256, 1,024).
SIZES = [(1, 1), (31, 33), (33, 64), (127, 65), (129, 257), (255, 255), (513, 1023), (2047, 1025),
         (2049, 2048), (4100, 2049), (9001, 4097), (70001, 300)]


@pytest.fixture(scope="module")
def ctx():
    with aidw.Context(0) as c:
        yield c


@pytest.mark.parametrize("precision", [aidw.F32C, aidw.F64, aidw.F64X])
@pytest.mark.parametrize("size", SIZES, ids=lambda s: f"n{s[0]}m{s[1]}")
def test_planned_and_forced_splits_match_the_oracle(ctx, precision, size):
    n, m = size
    wl = workloads.small_case(n + m, n, m, k=min(n, 5), pattern="uniform", side=50.0)
    ref, _ = oracle_for(wl, precision)
    tol = TOL_F32 if precision == aidw.F32C else TOL_F64
    ds = ctx.create_dataset(wl.x, wl.y, wl.z, wl.area)
    qx, qy = to_device(wl, precision)
    p = params_of(wl, precision)
    for splits in (0, 1, 3, 17, 70, 512):
        z = ctx.interpolate(ds, qx, qy, p, splits=(0, splits) if splits else None)[0]
        assert rel_err(z.cpu().numpy().astype(np.float64), ref).max() <= tol, splits
    assert ctx.check_device_errors() == aidw.OK
    ds.destroy()


def test_a_budget_below_the_planned_partial_sums_takes_fewer_splits():
    """8,192 queries plan about 20 MiB of partial sums; a context with 4 MiB left answers with
    fewer splits."""
    wl = workloads.small_case(5, 40000, 8192, k=10, pattern="uniform", side=50.0)
    ref, _ = oracle_for(wl, aidw.F32C)
    with aidw.Context(0, hbm_budget=8 << 20) as c:
        ds = c.create_dataset(wl.x, wl.y, wl.z, wl.area)
        qx, qy = to_device(wl, aidw.F32C)
        z = c.interpolate(ds, qx, qy, params_of(wl, aidw.F32C))[0]
        assert rel_err(z.cpu().numpy().astype(np.float64), ref).max() <= TOL_F32
        ds.destroy()


@pytest.mark.parametrize("precision", [aidw.F64, aidw.F64X])
@pytest.mark.parametrize("side", [1e-30, 1e-9, 1e9, 1e30])
def test_fp64_scales(ctx, precision, side):
    """The squared distances formed on the integer pipe, from far below to far above 1, with
    queries on data points and on one axis with them."""
    wl = workloads.small_case(9, 3001, 257, k=10, pattern="uniform", side=side)
    wl.qx[:20], wl.qy[:20] = wl.x[:20], wl.y[:20]
    wl.qx[20:40] = wl.x[20:40]
    ref, _ = oracle_for(wl, precision)
    ds = ctx.create_dataset(wl.x, wl.y, wl.z, wl.area)
    qx, qy = to_device(wl, precision)
    z = ctx.interpolate(ds, qx, qy, params_of(wl, precision))[0].cpu().numpy()
    assert rel_err(z, ref).max() <= TOL_F64
    ds.destroy()
