"""What admission charges for a served request covers what its launch takes, also where the request
runs phase 2 by power classes under a shape of more queries per thread: with the context's budget
filled to the byte by the admission budget, a request that is launched succeeds."""
import numpy as np
import pytest

from paper_1511_02186_gb300 import aidw, workloads

pytestmark = pytest.mark.gpu


def serve(wl, inflight, shape):
    """(launched, status) of one request with `inflight` bytes beside the dataset."""
    f4 = [np.asarray(v, dtype=np.float32) for v in (wl.x, wl.y, wl.z, wl.qx, wl.qy)]
    with aidw.Context(0) as big:
        d = big.create_dataset(*f4[:3], wl.area, dtype="f4")
        n, size = aidw.ctypes.c_int64(), aidw.ctypes.c_size_t()
        assert big.lib.aidw_dataset_info(big.ptr, d.handle, aidw.ctypes.byref(n),
                                         aidw.ctypes.byref(size)) == aidw.OK
        d.destroy()
    with aidw.Context(0, hbm_budget=size.value + inflight) as ctx:
        ctx.set_tune_config(shape)
        ds = ctx.create_dataset(*f4[:3], wl.area, dtype="f4")
        ctx.serving_configure(inflight_bytes=inflight)
        out = np.empty(wl.m, dtype=np.float32)
        status, rid = ctx.submit(ds, f4[3], f4[4], aidw.default_params(k=wl.k), out)
        assert status == aidw.OK
        status = ctx.wait(rid)
        launched = ctx.serving_stats().launches > 0
        ctx.release(rid)
        ds.destroy()
    return launched, status


@pytest.mark.parametrize("qpt", [2, 4, 8])
@pytest.mark.parametrize("m", [4095, 5000, 20000])
def test_least_admitted_budget_suffices(qpt, m):
    wl = workloads.small_case(97, 150001, m, k=10, pattern="uniform", side=100.0)
    shape = aidw.tune_config(queries_per_thread=qpt, split_points=4096)
    lo, hi = 1 << 16, 1 << 27
    assert serve(wl, hi, shape) == (True, aidw.OK)
    while hi - lo > 256:
        mid = (lo + hi) // 2
        launched, status = serve(wl, mid, shape)
        if launched:
            assert status == aidw.OK, f"launched with {mid} bytes, then {status}"
            hi = mid
        else:
            assert status == aidw.ERR_OOM
            lo = mid
