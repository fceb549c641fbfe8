"""cox_server_read: bounds, unknown tickets, and a compaction that keeps nothing or everything."""
import ctypes

import pytest

from tests.test_gpu_ops import cox  # noqa: F401 (a fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 5000, 100_003])
@pytest.mark.parametrize("d", [0.0, 1.0])
def test_read_bounds_and_counts(cox, n, d):  # noqa: F811
    import torch
    keys = torch.arange(n, dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    srv = cox.Server(64 << 20)
    try:
        for batch in (1, 3):  # alone (the op's own kernel), and in one launch
            reqs = [cox.make_request(cox.COX_REQ_COMPACT, keys, threshold=int(d * n)) for _ in range(batch)]
            tickets = srv.submit_many(reqs)
            for t, r in zip(tickets, reqs):
                srv.wait(t)
                got = srv.result(t, r)
                assert torch.equal(got, keys[:int(d * n)])
                room = ctypes.c_int64((4 * n + 255) // 256 * 64)  # words the output may hold
                dst = torch.empty(room.value + 64, dtype=torch.int32, device="cuda")
                read = cox.lib().cox_server_read
                assert read(srv.handle, t, dst.data_ptr(), room.value + 1, None) == cox.COX_EINVAL
                assert read(srv.handle, t, dst.data_ptr(), -1, None) == cox.COX_EINVAL
                assert read(srv.handle, t, None, 1, None) == cox.COX_EINVAL
                assert read(srv.handle, t, None, 0, None) == cox.COX_OK
                assert read(srv.handle, t + 1000, dst.data_ptr(), 1, None) == cox.COX_EINVAL
                torch.cuda.synchronize()
                srv.release(t)
                assert read(srv.handle, t, dst.data_ptr(), 1, None) == cox.COX_EINVAL
    finally:
        srv.close()
    assert cox.device_status() == cox.COX_OK
