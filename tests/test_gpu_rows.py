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
