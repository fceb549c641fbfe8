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
