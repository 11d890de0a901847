"""Calls one after the other on one stream without a wait between them, the queries rewritten in place
by another kernel before each: every call sees its own queries and leaves the results of a call made
alone, bit for bit (the kernels of a call, and of two calls, overlap at their ends)."""
import pytest

from paper_1511_02186_gb300 import aidw, workloads
from parity import is_f64

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [aidw.F32C, aidw.F64, aidw.F64X])
@pytest.mark.parametrize("m,splits", [(33, None), (1000, None), (5000, None), (1000, (3, 0)),
                                      (3000, (-2, 0))])
def test_queries_rewritten_between_calls(precision, m, splits):
    import torch
    rounds = 12
    wl = workloads.small_case(95, 20011, m, k=10, pattern="clustered", side=100.0)
    dt = torch.float64 if is_f64(precision) else torch.float32
    g = torch.Generator(device="cuda").manual_seed(7)
    qs = torch.rand((rounds, 2, m), generator=g, device="cuda", dtype=dt) * 100.0
    p = aidw.default_params(k=10, precision=precision)
    with aidw.Context(0) as ctx:
        ds = ctx.create_dataset(wl.x, wl.y, wl.z, wl.area)

        def call(qx, qy):
            return ctx.interpolate(ds, qx, qy, p, want_alpha=True, want_knn=True, splits=splits)

        alone = []
        for r in range(rounds):
            res = call(qs[r, 0], qs[r, 1])
            torch.cuda.synchronize()
            alone.append([t.clone() for t in res])
        torch.cuda.synchronize()
        for stream in (torch.cuda.current_stream(), torch.cuda.Stream()):
            with torch.cuda.stream(stream):
                qx, qy = (torch.empty(m, dtype=dt, device="cuda") for _ in range(2))
                got = []
                for r in range(rounds):
                    torch.mul(qs[r, 0], 1.0, out=qx)
                    torch.mul(qs[r, 1], 1.0, out=qy)
                    got.append(call(qx, qy))
            torch.cuda.synchronize()
            for a, b in zip(alone, got):
                for u, v in zip(a, b):
                    assert torch.equal(u, v)
        assert ctx.check_device_errors() == aidw.OK
        ds.destroy()
