"""Device memory of destroyed datasets: kept for the context's next calls up to a bound, never beyond
what the budget leaves beside the memory in use, and given back at shutdown."""
import numpy as np
import pytest

from paper_1511_02186_gb300 import aidw

pytestmark = pytest.mark.gpu

MIB = 1 << 20


def create(ctx, n):
    a = np.random.default_rng(1).uniform(0, 1, n).astype(np.float32)
    return ctx.create_dataset(a, a, a, 1.0, dtype="f4")


def test_budget_covers_what_destroyed_datasets_leave():
    """Six datasets of 58 MB in a budget of 400 MiB, destroyed; then one of 290 MB, which does not come
    from the pool: the context holds no more than its budget (and its temporary blocks) allows."""
    import torch
    torch.cuda.init()
    torch.cuda.synchronize()
    with aidw.Context(0, hbm_budget=400 * MIB) as ctx:
        free0 = torch.cuda.mem_get_info()[0]
        for ds in [create(ctx, 1_000_000) for _ in range(6)]:
            ds.destroy()
        big = create(ctx, 5_000_000)
        held = free0 - torch.cuda.mem_get_info()[0]
        assert held <= 400 * MIB + 8 * MIB, held / MIB
        big.destroy()
        again = [create(ctx, 1_000_000) for _ in range(6)]  # and it still serves the next ones
        for ds in again:
            ds.destroy()
        assert free0 - torch.cuda.mem_get_info()[0] <= 408 * MIB


def test_idle_memory_is_bounded_without_a_budget():
    import torch
    torch.cuda.init()
    torch.cuda.synchronize()
    with aidw.Context(0) as ctx:
        free0 = torch.cuda.mem_get_info()[0]
        for ds in [create(ctx, 1_000_000) for _ in range(40)]:  # 2.3 GB
            ds.destroy()
        assert free0 - torch.cuda.mem_get_info()[0] <= 1024 * MIB + 64 * MIB
    assert free0 - torch.cuda.mem_get_info()[0] <= 64 * MIB
