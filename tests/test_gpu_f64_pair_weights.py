"""Single weights of the FP64 phase 2 through the public call: four data points, three of them at one
place, give Z = r / (3 + r) with r = (D^2 / d^2)^(-power / 2), against decimal arithmetic. The far
point stands where the scan forms its squared distance on the FP64 pipe (index 1) or on the integer
pipe (index 3); powers from 2^-60 to 2^40, distances at very unequal dx and dy, near the smallest
and the largest doubles, and one nearly equal to the other."""
from decimal import Decimal, getcontext

import numpy as np
import pytest

from paper_1511_02186_gb300 import aidw

pytestmark = pytest.mark.gpu

getcontext().prec = 60

# (near dx, dy), (far dx, dy); the query is at 0.
PAIRS = [((0.3, 0.4), (0.3, 0.4000000001)), ((0.3, 0.4), (3.0, 4.0)), ((1.0, 0.0), (0.0, 1.5)),
         ((1.0, 1e-9), (1.0, 1e-7)), ((1e-20, 1.0), (1.7, 1e-300)), ((3.0, 1e-12), (1e3, 1e-9)),
         ((1e-30, 2e-30), (1e30, 3e29)), ((2e-38, 0.0), (0.0, 3e38)), ((5e-150, 1e-150), (7e-150, 0.0)),
         ((3e-153, 1e-153), (4e-153, 3e-153)), ((1e-120, 1e-200), (2e-120, 1e-121)),
         ((0.7, 0.1), (0.1, np.nextafter(0.7, 1.0)))]
POWERS = [2.0 ** -60, 1e-9, 0.3, 0.5, 0.9999, 1.0, 2.0, 2.5, 5.0, 31.7, 1e3, 1e6, 2.0 ** 40]


@pytest.mark.parametrize("far", [1, 3])
def test_weights(far):
    import torch
    with aidw.Context(0) as ctx:
        q = torch.zeros(1, dtype=torch.float64, device="cuda")
        for near, out in PAIRS:
            x, y, z = np.full(4, near[0]), np.full(4, near[1]), np.zeros(4)
            x[far], y[far], z[far] = out[0], out[1], 1.0
            ds = ctx.create_dataset(x, y, z, 1.0)
            d2, D2 = (Decimal(float(v[0])) ** 2 + Decimal(float(v[1])) ** 2 for v in (near, out))
            log_ratio = (D2 / d2).ln()
            for power in POWERS:
                got = ctx.idw(ds, q, q, power, aidw.F64).cpu().item()
                kappa = power / 2
                r = (-Decimal(kappa) * log_ratio).exp()
                want = r / (3 + r)
                # log2 of either square within 2^-52 of the square's own rounding (2^-52), times
                # kappa; the weight, the sums and the ratio to a few units in the last place.
                tol = Decimal((4 * kappa + 8) * 2.0 ** -52) * want + Decimal(1e-300)
                assert abs(Decimal(got) - want) <= tol, (near, out, power, got, want)
            ds.destroy()


@pytest.mark.parametrize("far", [1, 3])
def test_coincidence_and_overflow(far):
    """A query on the near points takes their value whatever is how near; a far point whose square is
    beyond a double has weight 0."""
    import torch
    with aidw.Context(0) as ctx:
        q = torch.zeros(1, dtype=torch.float64, device="cuda")
        for near, out, power in (((0.0, 0.0), (1e-150, 0.0), 1.0), ((0.0, 0.0), (1e-30, 2e-30), 0.5)):
            x, y, z = np.full(4, near[0]), np.full(4, near[1]), np.full(4, 2.5)
            x[far], y[far], z[far] = out[0], out[1], 1e6
            ds = ctx.create_dataset(x, y, z, 1.0)
            assert ctx.idw(ds, q, q, power, aidw.F64).cpu().item() == 2.5
            ds.destroy()
        x = np.array([1e30, 1.0, 1.0, 1.0])
        ds = ctx.create_dataset(x, x * 0.0, np.arange(4.0), 1.0)
        big = torch.tensor([1e200], dtype=torch.float64, device="cuda")
        assert np.isnan(ctx.idw(ds, big, big, 1.0, aidw.F64).cpu().item())
        ds.destroy()
