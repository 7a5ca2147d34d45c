"""The trainer's host copy of a batch: any source that numpy assignment takes, the same bits."""
import numpy as np
import pytest
import torch

from paper_2410_11625_gb300 import flnr_train

SHAPE = (3, 5, 40, 64)  # above the size at which torch splits a copy


def _base():
    a = np.random.default_rng(0).standard_normal(SHAPE).astype(np.float32)
    a[0, 0, 0, :4] = [np.nan, np.inf, -np.inf, -0.0]
    return a


def _unaligned(a):
    raw = np.zeros(a.nbytes + 1, np.uint8)
    v = raw[1:].view(np.float32).reshape(a.shape)
    v[...] = a
    return v


def _read_only(a):
    a.setflags(write=False)
    return a


@pytest.mark.parametrize("form", [
    lambda a: a, lambda a: a[:, :, ::-1, ::-1], lambda a: a.transpose(0, 1, 3, 2).copy().transpose(0, 1, 3, 2),
    lambda a: a[:1], lambda a: a.astype(np.float64), lambda a: a.astype(">f4"), _unaligned, _read_only,
    lambda a: a[:, :, :1], lambda a: torch.from_numpy(a), lambda a: np.float32(2.5)],
    ids=["plain", "flipped", "strided", "broadcast_batch", "float64", "big_endian", "unaligned", "read_only",
         "broadcast_rows", "tensor", "scalar"])
def test_fill_equals_assignment(form):
    src = form(_base())
    want = np.empty(SHAPE, np.float32)
    want[...] = src
    host = torch.full(SHAPE, 7.0)
    flnr_train._fill(host, src)
    assert np.array_equal(host.numpy().view(np.int32), want.view(np.int32))


def test_fill_refuses_what_assignment_refuses():
    with pytest.raises(ValueError):
        flnr_train._fill(torch.empty(SHAPE), np.zeros((3, 5, 40, 63), np.float32))
