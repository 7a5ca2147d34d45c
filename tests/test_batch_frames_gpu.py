"""The frame tables of the batch calls: the addresses of the tensors, None for no map guide, and the
errors that a wrong tensor gives in each place."""
import pytest

from test_flr_fast_gpu import flr  # noqa: F401

pytestmark = pytest.mark.gpu


def test_frame_table_addresses_and_errors(flr):  # noqa: F811
    import torch
    f = flr.FastFLR(q=4, factor=4, scale=2)
    d = flr.FLR(q=4, radius=2)
    g, y = torch.rand((4, 16, 24), device="cuda"), torch.rand((3, 16, 24), device="cuda")
    z, o = torch.rand((4, 32, 48), device="cuda"), torch.zeros((3, 32, 48), device="cuda")
    arr = f._frames([(g, y, z, o), (g, y, None, o)])
    assert (arr[0].guide, arr[0].radiance, arr[0].map_guide, arr[0].out) == (g.data_ptr(), y.data_ptr(), z.data_ptr(), o.data_ptr())
    assert arr[1].map_guide is None and (arr[1].H, arr[1].W) == (16, 24)
    frame = [g, y, z, o]
    bad = {"shape": lambda t: t[:, :-1].contiguous(), "channels": lambda t: t[:-1].contiguous(), "type": lambda t: t.double(),
           "stride": lambda t: t.transpose(1, 2).contiguous().transpose(1, 2), "host": lambda t: t.cpu(), "none": lambda t: None}
    for call, same, shapes in ((f.denoise_batch, False, ValueError), (d.denoise_batch, True, ValueError)):
        good = [g, y, g, torch.zeros_like(y)] if same else frame
        for k in range(4):
            for name, change in bad.items():
                if (name, k) == ("none", 2):
                    continue
                args = list(good)
                args[k] = change(args[k])
                with pytest.raises((TypeError, shapes, AttributeError)):
                    call([tuple(args)])
    f.denoise_batch([tuple(frame)])
    assert f.batch_status() == 0 and bool(torch.isfinite(o).all())
    f.close()
    d.close()
