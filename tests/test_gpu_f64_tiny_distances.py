"""FP64 and FP64X where squared distances approach the smallest normal double: every coordinate and
the area scaled by powers of two (exact, and Z does not depend on the scale), against the oracle on
the unscaled points."""
import numpy as np
import pytest

from paper_1511_02186_gb300 import aidw, workloads
from parity import TOL_F64, oracle_for, params_of, rel_err

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [aidw.F64, aidw.F64X])
@pytest.mark.parametrize("exponent", [0, -440, -470, -485, -500])
@pytest.mark.parametrize("m", [300, 2500])
def test_scaled_coordinates(precision, exponent, m):
    """Squared distances from about 2^-1012 on; m on both sides of the point-group kernel."""
    import torch
    wl = workloads.small_case(91, 4001, m, k=10, pattern="uniform", side=64.0)
    ref, _ = oracle_for(wl, precision)
    s = 2.0 ** exponent
    d1 = ((wl.qx[:, None] - wl.x) ** 2 + (wl.qy[:, None] - wl.y) ** 2).min()
    assert d1 * s * s > 2.0 ** -1020
    with aidw.Context(0) as ctx:
        ds = ctx.create_dataset(wl.x * s, wl.y * s, wl.z, wl.area * s * s)
        qx, qy = (torch.as_tensor(v * s, device="cuda") for v in (wl.qx, wl.qy))
        z, a, kn = ctx.interpolate(ds, qx, qy, params_of(wl, precision), want_alpha=True,
                                   want_knn=True)
        ds.destroy()
    assert rel_err(z.cpu().numpy(), ref).max() <= TOL_F64
    assert np.abs(a.cpu().numpy() - ref["alpha"]).max() <= 1e-6
    assert np.array_equal(kn.cpu().numpy(), ref["knn"])
