"""Device memory of a network for a small frame: its partial weight gradients are as many slices as
launches write (a third of the SMs' for the layers split over three columns of taps), 48 MB, and
the rest is below 4 MB; every allocation may be rounded up to 2 MiB."""
import pytest

from paper_2410_11625_gb300 import flnr

pytestmark = pytest.mark.gpu


def test_partials_are_as_large_as_the_launches_need():
    import torch
    torch.zeros(1, device="cuda")
    weights = flnr.init_weights(3)
    flnr.FLNR(64, weights).close()  # the library's own first allocations
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    net = flnr.FLNR(64, weights)
    used = before - torch.cuda.mem_get_info()[0]
    net.close()
    n_sm = torch.cuda.get_device_properties(0).multi_processor_count
    slices = 0
    for _, cin, cout, k in flnr.LAYERS:
        ci, co = -(-cin // 16) * 16, -(-cout // 16) * 16
        slices += max(1, n_sm // (3 if k * k * ci > 512 else 1)) * co * (k * k * ci + 8) * 4
    print(f"{used / 1e6:.1f} MB for {slices / 1e6:.1f} MB of slices")
    assert used <= slices + 4e6 + 4 * 2 ** 21
