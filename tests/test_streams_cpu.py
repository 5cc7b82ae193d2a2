"""The stream a product's outputs belong to: a call on a stream of the caller's returns the buffers that the library
wrote (a copy would be queued on torch's current stream, behind which nothing on the caller's stream waits); a call on
torch's current stream returns finished copies.  The library is a stand-in on host memory."""
import ctypes
from types import SimpleNamespace

import numpy as np
import pytest
import torch

from paper_1004_4548_gb300 import binding

N = 3            # terms of every product
CURRENT = 11     # torch's current stream


class Library:
    def __init__(self, coef):
        self.coef = coef

    def _mul(self, ctx, f, g, h, opts, stream):
        h = h._obj
        self.capacity, self.coef_ptr, self.stream = h.capacity, h.coef, stream
        h.nterms = N
        ctypes.memmove(h.coef, self.coef.ctypes.data, self.coef.nbytes)
        return binding.KR_OK

    poly_mul = poisson_mul = _mul


def product(monkeypatch, kind, stream):
    done = []
    monkeypatch.setattr(binding, "_alloc", lambda shape, dt, dev, host: torch.zeros(shape, dtype=getattr(torch, np.dtype(dt).name)))
    monkeypatch.setattr(binding, "_stream_ptr", lambda s: CURRENT if s is None else s)
    monkeypatch.setattr(binding, "_copies_done", done.append)
    lib = Library(np.arange(1, N + 1, dtype=np.int64 if kind == "poly" else np.float64))
    ctx = SimpleNamespace(L=lib, h=None, device=0)
    n = 20000
    e = torch.zeros((3, n), dtype=torch.int32)
    if kind == "poly":
        c = torch.zeros(n, dtype=torch.int64)
        coef = binding.poly_mul(e, c, e, c, ctx=ctx, stream=stream)[1]
    else:
        p = SimpleNamespace(exps=e, trig=e, kind=torch.zeros(n, dtype=torch.uint8), coef=torch.zeros(n, dtype=torch.float64))
        coef = binding.poisson_mul(p, p, ctx=ctx, stream=stream)[3]
    assert coef.tolist() == [1, 2, 3]
    return lib, coef, done


@pytest.mark.parametrize("kind", ["poly", "poisson"])
def test_callers_stream(monkeypatch, kind):
    lib, coef, done = product(monkeypatch, kind, 5)
    assert lib.stream == 5 and coef.data_ptr() == lib.coef_ptr and not done
    assert lib.capacity <= 80000   # what is returned keeps no more room alive than the operands' lengths suggest


@pytest.mark.parametrize("kind", ["poly", "poisson"])
@pytest.mark.parametrize("stream", [None, CURRENT])
def test_current_stream(monkeypatch, kind, stream):
    lib, coef, done = product(monkeypatch, kind, stream)
    assert lib.stream == CURRENT and coef.data_ptr() != lib.coef_ptr
    assert len(done) == 1 and done[0].data_ptr() == coef.data_ptr()   # the copies are waited for
