"""The C library is loaded once, and every thread that comes early gets that object with its
functions' types set (without types ctypes passes an address as a 32-bit integer).  The load is
slowed down, so that the threads meet in it."""
import ctypes
import threading
import time

import __graft_entry__
from paper_2410_11625_gb300 import flnr, flr


def test_one_library_object_with_types(monkeypatch):
    __graft_entry__.build()
    loads = []

    class Slow(ctypes.CDLL):
        def __init__(self, *a, **k):
            super().__init__(*a, **k)
            loads.append(self)
            time.sleep(0.05)

    monkeypatch.setattr(flr.ctypes, "CDLL", Slow)
    monkeypatch.setattr(flr, "_lib", None)
    monkeypatch.setattr(flnr, "_bound", False)
    start, got, bad = threading.Barrier(8), [], []

    def run(k):
        start.wait()
        time.sleep(0.02 * (k % 3))
        lib = flnr._lib() if k % 2 else flr.load_library()
        if lib.flr_denoise.argtypes is None or (k % 2 and lib.flnr_set_weights.argtypes is None):
            bad.append(k)
        got.append(lib)

    threads = [threading.Thread(target=run, args=(k,)) for k in range(8)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert len(got) == 8 and not bad
    assert len(loads) == 1 and all(lib is got[0] for lib in got)
    assert flnr._lib() is got[0] and got[0].flnr_set_weights.argtypes is not None
