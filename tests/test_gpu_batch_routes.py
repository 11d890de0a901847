"""Batch items in a batch whose queries fill the GPU (pruned phase-1 units where the queries are dense)
and alone (one query per warp): the same bits, and the oracle's values."""
import numpy as np
import pytest

from paper_1511_02186_gb300 import aidw, workloads
from parity import TOL_F32, oracle_for, params_of, rel_err, to_device

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,m,k", [(5001, 1024, 10), (5000, 1023, 10), (8000, 4096, 15),
                                   (20011, 4093, 6), (20011, 4003, 16), (3001, 8191, 32)])
def test_item_alone_and_in_a_batch_that_fills_the_gpu(n, m, k):
    import torch
    count = 200000 // m + 2
    wl = workloads.small_case(98, n, m, k=k, pattern="clustered", side=100.0)
    with aidw.Context(0) as ctx:
        ds = ctx.create_dataset(wl.x, wl.y, wl.z, wl.area)
        qx, qy = to_device(wl, aidw.F32C)
        p = params_of(wl, aidw.F32C)

        def items(c):
            return [(ds, qx, qy, p, torch.full((m,), float("nan"), device="cuda"),
                     torch.full((m,), float("nan"), device="cuda")) for _ in range(c)]

        alone, mixed = items(1), items(count)
        ctx.interpolate_batch(alone)
        ctx.interpolate_batch(mixed)
        torch.cuda.synchronize()
        assert ctx.check_device_errors() == aidw.OK
        for it in mixed:
            assert torch.equal(it[4], alone[0][4]) and torch.equal(it[5], alone[0][5])
        ref, _ = oracle_for(wl, aidw.F32C)
        z = alone[0][4].cpu().numpy().astype(np.float64)
        assert rel_err(z, ref).max() <= TOL_F32
        ds.destroy()
