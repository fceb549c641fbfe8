"""The tile pipeline when a wait runs out: every warp stops, nothing wrong is written, the library works on."""
import numpy as np
import pytest

from paper_2112_10034_gb300 import inputs
from tests.test_gpu_ops import POISON, cox, poisoned  # noqa: F401 (cox is a fixture)

pytestmark = pytest.mark.gpu
TILE = 8192
THR = 2**30


def _withheld_call(cox, k, tile, limit):  # noqa: F811
    """A compaction whose descriptor of `tile` stays withheld (both flag bits
    set: descriptors only grow).  Returns (out, count, seconds)."""
    import torch
    n = k.numel()
    out = poisoned(n, torch.int32)
    cnt = torch.full((1,), -1, dtype=torch.int64, device="cuda")
    ws_bytes = cox.cox_ballot_compact_workspace(n, 256)
    ws = torch.zeros(ws_bytes // 8, dtype=torch.int64, device="cuda")
    ws[256 // 8 + tile] = -(1 << 62)
    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    cox.cox_set_spin_limit(limit)
    try:
        a.record()
        assert cox.cox_ballot_compact(cox.COX_I32, 32, 256, k.data_ptr(), n, THR, out.data_ptr(), cnt.data_ptr(),
                                      ws.data_ptr(), ws_bytes, cox.COX_F_WS_READY, None) == cox.COX_OK
        b.record()
        assert cox.device_status() == cox.COX_ETIMEOUT
    finally:
        cox.cox_set_spin_limit(0)
    assert cox.device_status() == cox.COX_OK  # the word was cleared
    return out, cnt, a.elapsed_time(b) * 1e-3


def _keys(n):
    import torch
    return torch.from_numpy(inputs.uniform_u31(n, seed=n)).cuda()


def _tiles(short):
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    return 8 if short else 13 * sms  # one CTA per tile up to six per SM, then the pipeline


@pytest.mark.parametrize("short", [True, False])
@pytest.mark.parametrize("where", ["first", "middle", "last but one"])
def test_a_withheld_count_stops_the_tiles_after_it(cox, short, where):  # noqa: F811
    import torch
    t = _tiles(short)
    k = _keys(t * TILE - 5)
    tile = {"first": 0, "middle": t // 2, "last but one": t - 2}[where]
    out, cnt, _ = _withheld_call(cox, k, tile, 1000)
    assert int(cnt.item()) == -1  # the last tile never had its prefix
    kept = k[k < THR]
    upto = int((k[:(tile + 1) * TILE] < THR).sum())  # the withheld tile's own prefix is known
    got = out[:upto]
    assert bool(((got == kept[:upto]) | (got == POISON)).all())
    assert bool((out[upto:] == POISON).all())
    got, c = cox.ballot_compact(k, THR)  # and the library still works
    assert int(c.item()) == kept.numel() and torch.equal(got[:kept.numel()], kept)
    assert cox.device_status() == cox.COX_OK


def test_the_pipeline_waits_for_as_many_polls_as_the_limit_says(cox):  # noqa: F811
    """A poll for a count reads memory, some 0.5 us or more: no warp of the CTA may
    give up long before the one that polls has used its polls."""
    polls = 20_000
    _, _, seconds = _withheld_call(cox, _keys(_tiles(False) * TILE), 0, polls)
    assert 0.25e-6 * polls <= seconds <= 1.0


@pytest.mark.parametrize("off", [0, 1])
def test_compaction_in_place_through_the_pipeline(cox, off):  # noqa: F811
    """A tile is read before anything is written over it."""
    import torch
    k = _keys(_tiles(False) * TILE + 77 + off)[off:]
    want = k[k < THR]
    _, c = cox.ballot_compact(k, THR, out=k)
    assert int(c.item()) == want.numel() and torch.equal(k[:want.numel()], want)
    assert cox.device_status() == cox.COX_OK


@pytest.mark.parametrize("excl", [False, True])
@pytest.mark.parametrize("delta", [-1, 0, 1])
@pytest.mark.parametrize("tiles", [1, 33, "most"])
def test_int_sums_around_the_short_forms_limit(cox, tiles, delta, excl):  # noqa: F811
    """In place: one tile per CTA up to 16 per SM, with groups of 32 tiles, then the pipeline."""
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n = (16 * sms if tiles == "most" else tiles) * TILE + delta
    x = torch.randint(-1000, 1000, (n,), dtype=torch.int32, device="cuda")
    want = x.long().cumsum(0) - (x if excl else 0)
    room = torch.full((cox.cox_scan_workspace(cox.COX_SCOPE_GRID, n) + 256,), 0xA5, dtype=torch.uint8, device="cuda")
    cox.scan(x, exclusive=excl, out=x, workspace=room[:-256])
    assert torch.equal(x, want.to(torch.int32))
    assert bool((room[-256:] == 0xA5).all())
    assert cox.device_status() == cox.COX_OK
