"""wd.Lattice.set_gauge on links that are not contiguous: the copy it hands to the library is alive during the call."""

import gc
import weakref

import torch

from paper_2602_14450_gb300 import wd


class Library:
    """Stands in for the C library: checks what the pointer of wd_set_gauge points at."""

    def __init__(self):
        self.copies = []
        self.alive = None

    def wd_set_gauge(self, handle, ptr, where):
        gc.collect()
        self.alive = [r() is not None and r().data_ptr() == ptr for r in self.copies]
        return wd.WD_OK


class Links(torch.Tensor):
    lib = None

    def contiguous(self):
        c = torch.Tensor.contiguous(self.as_subclass(torch.Tensor))
        Links.lib.copies.append(weakref.ref(c))
        return c


def test_copy_outlives_the_call(monkeypatch):
    Links.lib = library = Library()
    monkeypatch.setattr(wd, "lib", lambda: library)
    lat = wd.Lattice.__new__(wd.Lattice)
    lat.h = None
    u = torch.zeros(2, 18, 4, dtype=torch.float64).transpose(0, 2).as_subclass(Links)
    lat.set_gauge(u)
    assert library.alive == [True]
