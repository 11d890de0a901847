"""A dataset made from device arrays that another stream is still writing."""
import pytest

from paper_1511_02186_gb300 import aidw

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [2000, 300000])
@pytest.mark.parametrize("dtype", ["f4", "f8"])
def test_arrays_in_flight_on_another_stream(n, dtype):
    import torch
    dt = torch.float32 if dtype == "f4" else torch.float64
    g = torch.Generator(device="cuda").manual_seed(3)
    good = torch.rand((3, n), generator=g, device="cuda", dtype=dt)
    q = torch.rand((2, 500), generator=g, device="cuda", dtype=torch.float32)
    with aidw.Context(0) as ctx:
        def result(arrays):
            ds = ctx.create_dataset(*arrays, 1.0, dtype=dtype)
            z = ctx.interpolate(ds, q[0], q[1])[0]
            torch.cuda.synchronize()
            ds.destroy()
            return z

        want = result([good[i] for i in range(3)])
        side = torch.cuda.Stream()
        for _ in range(3):
            late = [torch.zeros(n, device="cuda", dtype=dt) for _ in range(3)]
            torch.cuda.synchronize()
            with torch.cuda.stream(side):
                torch.cuda._sleep(20_000_000)  # about 10 ms
                for t, v in zip(late, good):
                    t.copy_(v)
            assert torch.equal(result(late), want)
