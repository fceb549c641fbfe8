"""A spin limit of one poll: kernels may give up, but end in order, and the next call is right."""
import pytest

from tests.test_gpu_ops import POISON, cox, poisoned  # noqa: F401 (cox is a fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [100_000, 20_000_003])
def test_calls_end_and_the_next_ones_are_right(cox, n):  # noqa: F811
    import torch
    x = torch.randint(-1000, 1000, (n,), dtype=torch.int32, device="cuda")
    out = poisoned(n, torch.int32)
    cnt = torch.zeros(1, dtype=torch.int64, device="cuda")
    ws = torch.zeros(max(cox.cox_scan_workspace(cox.COX_SCOPE_GRID, n), cox.cox_ballot_compact_workspace(n, 256)),
                     dtype=torch.uint8, device="cuda")
    i32, xp, op, wp, wb = cox.COX_I32, x.data_ptr(), out.data_ptr(), ws.data_ptr(), ws.numel()
    calls = [lambda: cox.cox_tile_scan(0, i32, 32, 256, xp, op, n, 0, None),
             lambda: cox.cox_tile_reduce(0, i32, 8, 256, cox.COX_SCOPE_TILE, xp, op, n, 0, None, None, 0, None),
             lambda: cox.cox_scan(0, i32, cox.COX_SCOPE_BLOCK, 256, xp, op, n, 0, 0, None, 0, None),
             lambda: cox.cox_scan(0, i32, cox.COX_SCOPE_GRID, 256, xp, op, n, 0, 0, wp, wb, None),
             lambda: cox.cox_ballot_compact(i32, 32, 256, xp, n, 0, op, cnt.data_ptr(), wp, wb, 0, None)]
    for call in calls:
        cox.cox_set_spin_limit(1)
        try:
            assert call() == cox.COX_OK
            assert cox.device_status() in (cox.COX_OK, cox.COX_ETIMEOUT)
        finally:
            cox.cox_set_spin_limit(0)
        assert bool((out[n:] == POISON).all())
    assert cox.device_status() == cox.COX_OK
    assert torch.equal(cox.scan(x), x.long().cumsum(0).to(torch.int32))
    got, c = cox.ballot_compact(x, 0)
    assert torch.equal(got[:int(c.item())], x[x < 0])
    assert cox.device_status() == cox.COX_OK
