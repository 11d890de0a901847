"""Data at one location or a few: every distance of a query ties with its k-th, so no box and no point
can be left out by being farther. The result is exact, the neighbour lists are those of the
oracle's rule, and a call takes a few times as long as with spread data, not tens of times (the
scan must not take in every point of the tie)."""
import numpy as np
import pytest

from paper_1511_02186_gb300 import aidw
from parity import TOL_F32, TOL_F64, is_f64

pytestmark = pytest.mark.gpu


def make(n, m, locations, seed):
    rng = np.random.default_rng(seed)
    i = rng.integers(0, locations, n)
    px, py = rng.uniform(0.4, 0.6, locations), rng.uniform(0.4, 0.6, locations)
    z = rng.uniform(1.0, 2.0, n)
    return px[i], py[i], z, rng.uniform(0, 1, m), rng.uniform(0, 1, m), i


@pytest.mark.parametrize("precision", [aidw.F32C, aidw.F64, aidw.F64X])
@pytest.mark.parametrize("k", [1, 10, 32])
def test_results(precision, k):
    import torch
    n, m = 20003, 500
    x, y, z, qx, qy, _ = make(n, m, 1, 1)
    dt = torch.float64 if is_f64(precision) else torch.float32
    with aidw.Context(0) as ctx:
        ds = ctx.create_dataset(x, y, z, 1.0)
        q = [torch.as_tensor(v, dtype=dt, device="cuda") for v in (qx, qy)]
        out, _, kn = ctx.interpolate(ds, *q, aidw.default_params(k=k, precision=precision),
                                     want_knn=True)
        out, kn = out.cpu().numpy().astype(np.float64), kn.cpu().numpy()
        ds.destroy()
    want = (z if is_f64(precision) else z.astype(np.float32)).mean(dtype=np.float64)
    assert np.abs(out - want).max() / want <= (TOL_F64 if is_f64(precision) else TOL_F32)
    if is_f64(precision):
        assert (kn == np.arange(k)).all()  # ties to the lower index
    else:
        assert kn.min() >= 0 and kn.max() < n
        assert all(len(set(row)) == k for row in kn.tolist())


@pytest.mark.parametrize("precision,m,most", [(aidw.F32C, 8192, 20.0), (aidw.F64, 2048, 6.0),
                                              (aidw.F64X, 2048, 8.0)])
@pytest.mark.parametrize("locations", [1, 3])
def test_time(precision, m, most, locations):
    import torch
    n = 262144
    dt = torch.float64 if is_f64(precision) else torch.float32

    def best(ctx, places):
        x, y, z, qx, qy, _ = make(n, m, places, 2)
        ds = ctx.create_dataset(x, y, z, 1.0)
        q = [torch.as_tensor(v, dtype=dt, device="cuda") for v in (qx, qy)]
        p = aidw.default_params(precision=precision)
        times = []
        for _ in range(4):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            a.record()
            ctx.interpolate(ds, *q, p)
            b.record()
            torch.cuda.synchronize()
            times.append(a.elapsed_time(b))
        ds.destroy()
        return min(times[1:])

    with aidw.Context(0) as ctx:
        spread, tied = best(ctx, n), best(ctx, locations)
    assert tied <= most * spread, (tied, spread)
