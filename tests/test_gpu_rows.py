"""GPU parity of the row-per-lane streaming kernels where their launch shapes change."""
import numpy as np
import pytest

import oracle as o
from paper_2112_10034_gb300 import inputs
from tests.test_gpu_ops import cox, dev, host, poisoned  # noqa: F401 (cox is a fixture)

pytestmark = pytest.mark.gpu
POISON = 0x7FBADBAD
CHUNK = 1024  # elements of one warp chunk
WARPS = 8     # per CTA


@pytest.mark.parametrize("delta", [-CHUNK - 1, -1, 0, 1, CHUNK * WARPS + 33])
def test_compensated_tile_scan_around_two_chunks_per_warp(cox, delta):  # noqa: F811
    """Below 4 CTAs' worth of chunks per SM every warp takes one chunk, from there on two."""
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n = 4 * WARPS * sms * CHUNK + delta
    x = inputs.normal_f32(n, seed=7)
    xd, out = dev(x), poisoned(n, torch.float32)
    assert cox.cox_tile_scan(o.SUM, o.F32, 16, 256, xd.data_ptr(), out.data_ptr(), n, 1, None) == cox.COX_OK
    got = host(out)
    assert (got[n:].view(np.int32) == POISON).all()
    want = o.scan_emulate(o.SUM, o.F32, 16, 256, x, compensated=True)
    assert np.array_equal(got[:n].view(np.int32), want.view(np.int32))


@pytest.mark.parametrize("B", [32, 96, 256, 320, 544, 1024])
@pytest.mark.parametrize("dt,op,comp", [(o.F32, o.SUM, 0), (o.F32, o.SUM, 1), (o.F32, o.MAX, 0), (o.I32, o.SUM, 0),
                                        (o.U32, o.MIN, 0)])
@pytest.mark.parametrize("tail", [-1, 0, 1, 37])
def test_block_scan_rows_equal_the_general_kernel(cox, B, dt, op, comp, tail):  # noqa: F811
    """An aligned array (rows kernel from 2^16 elements, 2^19 compensated) and
    the same values 4 bytes off (the general kernel) give the same bits."""
    import torch
    n = (1 << (19 if comp else 16)) + tail
    g = torch.Generator(device="cuda")
    g.manual_seed(n + B)
    x = torch.randn(n, generator=g, device="cuda").view(torch.int32)
    off = torch.empty(n + 1, dtype=torch.int32, device="cuda")
    off[1:] = x
    for excl in (0, 1):
        got = []
        for src in (x, off[1:]):
            out = poisoned(n, torch.int32)
            assert cox.cox_scan(op, dt, o.BLOCK, B, src.data_ptr(), out.data_ptr(), n, comp, excl, None, 0,
                                None) == cox.COX_OK
            got.append(out)
        assert torch.equal(got[0], got[1]) and bool((got[0][n:] == POISON).all())
    # in place
    y = x.clone()
    assert cox.cox_scan(op, dt, o.BLOCK, B, y.data_ptr(), y.data_ptr(), n, comp, 1, None, 0, None) == cox.COX_OK
    assert torch.equal(y, got[1][:n])


@pytest.mark.parametrize("B", [32, 64, 256, 544, 1024])
@pytest.mark.parametrize("dt,op", [(o.F32, o.SUM), (o.F32, o.MIN), (o.I32, o.SUM)])
@pytest.mark.parametrize("delta", [-1, 0, 1, 37])
def test_block_scan_at_the_rows_kernels_smallest_sizes(cox, B, dt, op, delta):  # noqa: F811
    import torch
    n = (3 << (15 if B < 64 else 17)) + delta
    g = torch.Generator(device="cuda")
    g.manual_seed(n + B)
    off = torch.randn(n + 1, generator=g, device="cuda").view(torch.int32)[1:]
    x = off.clone()
    for excl in (0, 1):
        got = [poisoned(n, torch.int32) for _ in range(2)]
        for src, out in zip((x, off), got):
            assert cox.cox_scan(op, dt, o.BLOCK, B, src.data_ptr(), out.data_ptr(), n, 0, excl, None, 0,
                                None) == cox.COX_OK
        assert torch.equal(got[0], got[1]) and bool((got[0][n:] == POISON).all())


def _grid_scan(cox, src, n, op, dt, comp, excl):  # noqa: F811
    import torch
    out = poisoned(n, torch.int32)
    ws = torch.full((cox.cox_scan_workspace(o.GRID, n),), 0xA5, dtype=torch.uint8, device="cuda")
    assert cox.cox_scan(op, dt, o.GRID, 256, src.data_ptr(), out.data_ptr(), n, comp, excl, ws.data_ptr(), ws.numel(),
                        None) == cox.COX_OK
    assert bool((out[n:] == POISON).all())
    return out[:n]


GRID_TILE = {0: 6144, 1: 8192}  # elements per tile of the pipeline: 32-bit values, compensated pairs
GRID_BUFS = {0: 9, 1: 6}        # tiles a CTA keeps
SHORT_TILE = 8192               # of the short form, eight per SM at most


@pytest.mark.parametrize("where", ["row", "tile", "short", "buffers"])
@pytest.mark.parametrize("delta", [-33, -1, 0, 1, 32])
@pytest.mark.parametrize("dt,op,comp", [(o.I32, o.SUM, 0), (o.U32, o.MAX, 0), (o.I32, o.XOR, 0), (o.F32, o.MIN, 0),
                                        (o.F32, o.SUM, 1)])
def test_grid_scan_pipeline_equals_the_general_kernel(cox, where, delta, dt, op, comp):  # noqa: F811
    """Aligned arrays (the short form, the tile pipeline) against the same values 4 bytes off
    (the general kernel): whole numbers bit for bit, compensated sums to one
    rounding of the output (2^-24) on either side."""
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    t = GRID_TILE[comp]
    n = {"row": 64, "tile": 3 * SHORT_TILE, "short": 8 * sms * SHORT_TILE,
         "buffers": sms * (GRID_BUFS[comp] + 4) * t}[where] + delta
    g = torch.Generator(device="cuda")
    g.manual_seed(n + op)
    x = torch.randn(n, generator=g, device="cuda").view(torch.int32) if dt == o.F32 else \
        torch.randint(-2**31, 2**31 - 1, (n,), generator=g, device="cuda", dtype=torch.int32)
    off = torch.empty(n + 1, dtype=torch.int32, device="cuda")
    off[1:] = x
    for excl in (0, 1):
        a = _grid_scan(cox, x, n, op, dt, comp, excl)
        b = _grid_scan(cox, off[1:], n, op, dt, comp, excl)
        if comp:
            fa, fb = a.view(torch.float32).double(), b.view(torch.float32).double()
            # each is within u |y| + 2^-40 sum|x| of the exact prefix
            assert bool(((fa - fb).abs() <= 2.0**-23 * fb.abs() + 2.0**-39 * x.view(torch.float32).abs().sum()).all())
        else:
            assert torch.equal(a, b)
    assert cox.device_status() == cox.COX_OK


def test_grid_scan_is_reproducible_and_works_in_place(cox):  # noqa: F811
    """The running prefix is one sequence of combines; a tile is read before it is written."""
    import torch
    n = 3_000_017
    g = torch.Generator(device="cuda")
    g.manual_seed(5)
    x = torch.randint(-1000, 1000, (n,), generator=g, device="cuda", dtype=torch.int32)
    want = x.cumsum(0, dtype=torch.int64).to(torch.int32)
    ws = torch.empty(cox.cox_scan_workspace(o.GRID, n), dtype=torch.uint8, device="cuda")
    assert cox.cox_scan(o.SUM, o.I32, o.GRID, 256, x.data_ptr(), x.data_ptr(), n, 0, 0, ws.data_ptr(), ws.numel(),
                        None) == cox.COX_OK
    assert torch.equal(x, want)


@pytest.mark.parametrize("d", [0.0, 0.3, 1.0])
@pytest.mark.parametrize("where,delta", [("tile", -1), ("tile", 0), ("tile", 1), ("short", 0), ("short", 1),
                                         ("buffers", -511), ("buffers", 3)])
def test_compaction_forms_agree(cox, where, delta, d):  # noqa: F811
    """One tile per CTA, the tile pipeline, and both from an unaligned address, against a plain filter."""
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n = {"tile": 3, "short": 6 * sms, "buffers": 13 * sms}[where] * 8192 + delta
    g = torch.Generator(device="cuda")
    g.manual_seed(n)
    full = torch.randint(-2**31, 2**31 - 1, (n + 1,), generator=g, device="cuda", dtype=torch.int32)
    thr = int(-2**31 + d * 2**32)
    for keys in (full[:n], full[1:]):
        for dt in (o.I32, o.U32):
            out = poisoned(n, torch.int32)
            cnt = torch.full((1,), -1, dtype=torch.int64, device="cuda")
            ws = torch.full((cox.cox_ballot_compact_workspace(n, 256),), 0xA5, dtype=torch.uint8, device="cuda")
            t = thr if dt == o.I32 else thr + 2**31
            assert cox.cox_ballot_compact(dt, 32, 256, keys.data_ptr(), n, t, out.data_ptr(), cnt.data_ptr(),
                                          ws.data_ptr(), ws.numel(), 0, None) == cox.COX_OK
            unsigned = keys.long() & 0xFFFFFFFF
            want = keys[(keys.long() if dt == o.I32 else unsigned) < t]
            assert int(cnt.item()) == want.numel() and torch.equal(out[:want.numel()], want)
            assert bool((out[n:] == POISON).all())
    assert cox.device_status() == cox.COX_OK


@pytest.mark.parametrize("off", [1, 2, 3])
@pytest.mark.parametrize("tiles", [1, 2, "pipe"])
@pytest.mark.parametrize("delta", [-1, 0, 1, 2, 3, 4])
def test_compaction_of_unaligned_arrays(cox, off, tiles, delta):  # noqa: F811
    """Tiles copied from the 16-byte boundary before them; the ends of the array."""
    import torch
    t = 7 * torch.cuda.get_device_properties(0).multi_processor_count if tiles == "pipe" else tiles
    n = t * 8192 + delta
    g = torch.Generator(device="cuda")
    g.manual_seed(n)
    keys = torch.randint(-2**31, 2**31 - 1, (n + off,), generator=g, device="cuda", dtype=torch.int32)[off:]
    assert keys.data_ptr() % 16 == 4 * off
    for where in ("apart", "in place"):
        want = keys[keys < 0]
        out = poisoned(n, torch.int32) if where == "apart" else keys
        _, cnt = cox.ballot_compact(keys, 0, out=out)
        assert int(cnt.item()) == want.numel() and torch.equal(out[:want.numel()], want)
        assert where == "in place" or bool((out[want.numel():] == POISON).all())
    assert cox.device_status() == cox.COX_OK


@pytest.mark.parametrize("n", [32, 100_003, 3_000_001, 30_000_007])
def test_compensated_grid_scan_takes_the_smaller_workspace(cox, n):  # noqa: F811
    """Half of cox_scan_workspace(): aggregates packed into one word each."""
    import torch
    def align(b):
        return (b + 255) // 256 * 256
    t = -(-n // 16384)
    need = 256 + align(4 * t) + 16 * t + 24 * (-(-t // 32))
    x = torch.from_numpy(inputs.normal_f32(n, seed=n)).cuda()
    ws = torch.full((max(need, cox.cox_scan_workspace(o.GRID, n)),), 0xA5, dtype=torch.uint8, device="cuda")
    out = poisoned(n, torch.float32)

    def call(bytes_, comp=1):
        return cox.cox_scan(o.SUM, o.F32, o.GRID, 256, x.data_ptr(), out.data_ptr(), n, comp, 0, ws.data_ptr(), bytes_,
                            None)
    assert call(need - 1) == cox.COX_ENOMEM
    assert call(cox.cox_scan_workspace(o.GRID, n) - 1, 0) == cox.COX_ENOMEM
    assert call(need) == cox.COX_OK
    want = x.double().cumsum(0)
    err = (out[:n].double() - want).abs() / torch.maximum(want.abs(), 2.0**-24 * x.double().abs().cumsum(0))
    assert float(err.max()) <= 1e-5
    assert bool((ws[need:] == 0xA5).all())


@pytest.mark.parametrize("W", [2, 8, 16, 32])
@pytest.mark.parametrize("per_warp", [1, 5, 7, 9])
@pytest.mark.parametrize("comp", [0, 1])
def test_tile_ops_around_the_waves_limits(cox, W, per_warp, comp):  # noqa: F811
    """A wave of resident warps, or CTAs handed out by the hardware: the same bits as
    the general kernels (the same values 4 bytes off)."""
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    edge = 2 * WARPS * sms * per_warp * CHUNK  # chunks of 32 rows per resident warp
    g = torch.Generator(device="cuda")
    g.manual_seed(W)
    off = torch.randn(edge + 66, generator=g, device="cuda")[1:]
    x = off.clone()
    for n in (edge, edge + 33):
        outs = []
        for src in (x, off):
            scan, red, lo = poisoned(n, torch.float32), poisoned(-(-n // W), torch.float32), poisoned(-(-n // W), torch.float32)
            assert cox.cox_tile_scan(o.SUM, o.F32, W, 256, src.data_ptr(), scan.data_ptr(), n, comp, None) == cox.COX_OK
            assert cox.cox_tile_reduce(o.SUM, o.F32, W, 256, o.TILE, src.data_ptr(), red.data_ptr(), n, comp,
                                       lo.data_ptr() if comp else None, None, 0, None) == cox.COX_OK
            outs.append([t.view(torch.int32) for t in (scan, red, lo)])
        for a, b in zip(*outs):
            assert torch.equal(a, b)
            assert bool((a[-64:] == POISON).all())
    assert cox.device_status() == cox.COX_OK


@pytest.mark.parametrize("kind", ["inf", "nan", "zeros", "tiny", "huge"])
def test_special_values_as_in_the_general_kernels(cox, kind):  # noqa: F811
    """Infinities, NaN, signed zeros, denormals and overflow: aligned arrays (rows kernels, short form and pipeline)
    give what the same values 4 bytes off give, NaN for NaN."""
    import torch

    def same(a, b):
        fa, fb = a.view(torch.float32), b.view(torch.float32)
        return bool(((a == b) | (fa.isnan() & fb.isnan())).all())
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    for n in (600_003, 10 * sms * SHORT_TILE + 5):
        g = torch.Generator(device="cuda")
        g.manual_seed(n)
        off = torch.randn(n + 1, generator=g, device="cuda")[1:]
        idx = torch.randint(0, n, (n // 5000,), generator=g, device="cuda")
        if kind == "inf":
            off[idx], off[idx // 2] = float("inf"), -float("inf")
        elif kind == "nan":
            off[idx], off[0] = float("nan"), float("nan")
        elif kind == "zeros":
            off.zero_()
            off[idx] = -0.0
            off[:2000] = -0.0
        else:
            off.mul_(1e-40 if kind == "tiny" else 3e38)
        x = off.clone()
        ws = torch.empty(cox.cox_scan_workspace(o.GRID, n), dtype=torch.uint8, device="cuda")
        for op, comp in ((o.SUM, 0), (o.SUM, 1), (o.MIN, 0), (o.MAX, 0)):
            outs = {}
            for at, src in (("on", x), ("off", off)):
                for B in (32, 256):
                    for excl in (0, 1):
                        out = poisoned(n, torch.int32)
                        assert cox.cox_scan(op, o.F32, o.BLOCK, B, src.data_ptr(), out.data_ptr(), n, comp, excl, None, 0,
                                            None) == cox.COX_OK
                        outs[at, B, excl] = out[:n]
                for W in (2, 32):
                    out = poisoned(n, torch.int32)
                    assert cox.cox_tile_scan(op, o.F32, W, 256, src.data_ptr(), out.data_ptr(), n, comp, None) == cox.COX_OK
                    outs[at, W] = out[:n]
                if op != o.SUM:  # (sums are folded in another order)
                    out = poisoned(n, torch.int32)
                    assert cox.cox_scan(op, o.F32, o.GRID, 256, src.data_ptr(), out.data_ptr(), n, 0, 0, ws.data_ptr(),
                                        ws.numel(), None) == cox.COX_OK
                    outs[at, "grid"] = out[:n]
            for key in [k for k in outs if k[0] == "on"]:
                assert same(outs[key], outs[("off",) + key[1:]]), (kind, n, op, comp, key)
    assert cox.device_status() == cox.COX_OK
