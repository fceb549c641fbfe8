"""The binding tells the library how large a caller's workspace is, not how large one should be."""
import pytest

from paper_2112_10034_gb300 import cox as c

OPS = {  # helper: (the C call it makes, its position of the size, the size the library asks for)
    "scan": ("cox_scan", 10, lambda x: c.cox_scan_workspace(c.COX_SCOPE_GRID, x.numel())),
    "tile_reduce": ("cox_tile_reduce", 11, lambda x: c.cox_tile_reduce_workspace(c.COX_SCOPE_GRID, x.numel(), 256)),
    "grid_broadcast": ("cox_grid_broadcast", 6, lambda x: c.cox_grid_broadcast_workspace(x.numel())),
}


def _call(helper, x, **kw):
    if helper != "grid_broadcast":
        kw["scope"] = c.COX_SCOPE_GRID
    return getattr(c, helper)(x, **kw)


@pytest.mark.parametrize("helper", OPS)
@pytest.mark.parametrize("dtype,count", [("uint8", 48), ("int64", 6), ("uint8", 1 << 20)])
def test_the_size_passed_is_the_tensors_own(helper, dtype, count, monkeypatch):
    import torch
    entry, at, _ = OPS[helper]
    seen = []
    monkeypatch.setattr(c, entry, lambda *a: seen.append(a[at]) or c.COX_OK)
    monkeypatch.setattr(c, "_dev_tensor", lambda x: x)
    monkeypatch.setattr(c, "_stream", lambda dev: 0)
    w = torch.empty(count, dtype=getattr(torch, dtype))
    _call(helper, torch.zeros(100_000), workspace=w)
    _call(helper, torch.zeros(100_000))
    assert seen == [w.numel() * w.element_size(), OPS[helper][2](torch.zeros(100_000))]


@pytest.mark.gpu
@pytest.mark.parametrize("helper", OPS)
def test_a_workspace_too_small_is_refused_and_left_alone(helper):
    import torch
    x = torch.randn(100_000, device="cuda")
    room = torch.full((OPS[helper][2](x) + 4096,), 0xA5, dtype=torch.uint8, device="cuda")
    with pytest.raises(c.CoxError) as e:
        _call(helper, x, workspace=room[:64])
    assert e.value.status == c.COX_ENOMEM
    assert bool((room == 0xA5).all())


@pytest.mark.gpu
@pytest.mark.parametrize("n", [100_003, 30_000_007])
def test_compensated_scan_stays_inside_the_smaller_workspace(n):
    """The size a compensated grid scan used with 16384-element tiles is still enough."""
    import torch
    t = -(-n // 16384)
    need = 256 + (4 * t + 255) // 256 * 256 + 16 * t + 24 * -(-t // 32)
    x = torch.randn(n, device="cuda")
    room = torch.full((c.cox_scan_workspace(c.COX_SCOPE_GRID, n),), 0xA5, dtype=torch.uint8, device="cuda")
    y = c.scan(x, compensated=True, workspace=room[:need]).double()
    want = x.double().cumsum(0)
    err = (y - want).abs() / torch.maximum(want.abs(), 2.0**-24 * x.double().abs().cumsum(0))
    assert float(err.max()) <= 1e-5
    assert bool((room[need:] == 0xA5).all())
