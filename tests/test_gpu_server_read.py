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


@pytest.mark.parametrize("side", [False, True])
def test_a_released_requests_memory_waits_for_its_copy(cox, side):  # noqa: F811
    """The copy is behind ordinary work on the caller's stream when its request is
    released; the next request needs the same memory (the budget holds one)."""
    import torch
    n = 1 << 22
    xs = [torch.randint(-1000, 1000, (n,), dtype=torch.int32, device="cuda") for _ in range(3)]
    reqs = [cox.make_request(cox.COX_REQ_SCAN, x, width=32) for x in xs]
    a = torch.randn(8192, 8192, device="cuda", dtype=torch.bfloat16)
    torch.cuda.synchronize()
    srv = cox.Server(10 * n)  # a request holds 4 n bytes of input and 4 n of output
    st = torch.cuda.Stream() if side else torch.cuda.current_stream()
    got = []
    with torch.cuda.stream(st):
        for r in reqs:
            t = srv.submit(r)
            srv.wait(t)
            for _ in range(20):  # some 10 ms
                a @ a
            got.append(srv.result(t, r))
            got.append(srv.result(t, r))  # (a request may be read more than once)
            srv.release(t)
        srv.close()  # the last copies may still be waiting
    torch.cuda.synchronize()
    for i, y in enumerate(got):
        want = xs[i // 2].view(-1, 32).cumsum(1, dtype=torch.int64).to(torch.int32).view(-1)
        assert torch.equal(y, want)


def test_released_memory_is_all_given_back(cox):  # noqa: F811
    """With copies out of order on two streams, and requests never read."""
    import torch
    x = torch.arange(50_000, dtype=torch.int32, device="cuda")
    a = torch.randn(4096, 4096, device="cuda", dtype=torch.bfloat16)
    torch.cuda.synchronize()
    srv = cox.Server(64 << 20)
    try:
        for _ in range(3):
            tickets = srv.submit_many([cox.make_request(cox.COX_REQ_SCAN, x, width=8) for _ in range(30)])
            slow = torch.cuda.Stream()
            r = cox.make_request(cox.COX_REQ_SCAN, x, width=8)
            for i, t in enumerate(tickets):
                srv.wait(t)
                if i % 3 == 0:
                    with torch.cuda.stream(slow):
                        a @ a
                        srv.result(t, r)
                elif i % 3 == 1:
                    srv.result(t, r)
                srv.release(t)
            torch.cuda.synchronize()
            assert srv.stats()["used_bytes"] == 0
    finally:
        srv.close()
