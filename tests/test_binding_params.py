"""peel_batch's parameters, marshalled (CPU; the library call is a stand-in that
keeps what it is given): any iterable of Params, subclasses among them, reaches
the library as the same bytes.
"""
import ctypes

import pytest

from paper_2504_09311_gb300 import dupin


class _Lib:
    def dupin_peel_batch(self, G, P, R, k, stream):
        self.got = ctypes.string_at(P, k * ctypes.sizeof(dupin.Params))
        return dupin.OK


class _Graph:
    n = 3
    handle = ctypes.c_void_p(8)


class _Own(dupin.Params):
    pass


@pytest.mark.parametrize("form", [list, tuple, iter, lambda p: (q for q in p), lambda p: map(lambda q: q, p),
                                  lambda p: (dupin.Params * len(p))(*p),
                                  lambda p: [_Own.from_buffer_copy(q) for q in p]])
def test_any_iterable_of_params(monkeypatch, form):
    lib = _Lib()
    monkeypatch.setattr(dupin, "lib", lambda: lib)
    monkeypatch.setattr(dupin, "_stream", lambda s: None)
    params = [dupin.make_params(m, k, (1, 10 + k)) for m in ("dg", "fd") for k in (1, 2, 3)]
    dupin.peel_batch([_Graph()] * len(params), form(params))
    assert lib.got == b"".join(map(bytes, params))
