"""The single-call tuner times a candidate shape only where the call runs other kernels under it: a call
whose phase 1 is one warp per query and whose phase 2 runs by power classes or point groups has one
shape, so the tuner runs it alone and returns the shape it started from."""
import pytest

from paper_1511_02186_gb300 import aidw, workloads
from parity import params_of, to_device

pytestmark = pytest.mark.gpu

START = dict(queries_per_thread=8, tile_points=256, knn_list=32)


def tune(n, m, levels, allocations, start=START):
    wl = workloads.small_case(99, n, m, k=10, pattern="uniform", side=100.0, levels=levels)
    with aidw.Context(0) as ctx:
        ctx.set_tune_config(aidw.tune_config(**start))
        ds = ctx.create_dataset(wl.x, wl.y, wl.z, wl.area)
        qx, qy = to_device(wl, aidw.F32C)
        ctx.fail_alloc_after(allocations)  # every run of the call allocates its scratch once
        cfg, ms, _ = ctx.autotune_interpolate(ds, qx, qy, params_of(wl, aidw.F32C), reps=2)
        ctx.fail_alloc_after(-1)
        ds.destroy()
    return cfg, ms


@pytest.mark.parametrize("n,m,levels", [(60000, 20000, (1, 2, 3, 4, 5)), (60000, 1000, (1, 2, 3, 4, 5)),
                                        (60000, 2048, (1, 1.5, 2, 2.5, 3.5))])
def test_calls_of_one_shape(n, m, levels):
    cfg, ms = tune(n, m, levels, 4)  # a warm-up, two timed runs, the last one
    assert cfg == aidw.tune_config(**START) and ms > 0


def test_a_call_with_several_shapes_is_searched():
    with pytest.raises(aidw.AidwError) as e:
        tune(60000, 20000, (1.2, 1.5, 2, 2.5, 3.5), 4)
    assert e.value.status == aidw.ERR_OOM
    cfg, ms = tune(60000, 20000, (1.2, 1.5, 2, 2.5, 3.5), 1000)
    assert aidw.tune_config_valid(cfg) and ms > 0
