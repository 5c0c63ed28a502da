"""Strided tensors as arguments: the contiguous copies made for a call have to live until it returns.
A stand-in for the library, on host tensors, reads its arguments' memory inside the call, where a
copy that was already released holds the next copy's values."""
import ctypes
from types import SimpleNamespace

import numpy as np
import pytest
import torch

import paper_2004_07732_gb300._lib as binding

N = 4096


def _strided(seed):
    """N complex numbers in every second place of a tensor, and their values"""
    g = torch.Generator().manual_seed(seed)
    t = torch.randn(2 * N, dtype=torch.complex128, generator=g)[::2]
    return t, t.numpy().copy()


def _values(address):
    address = address.value if isinstance(address, ctypes.c_void_p) else address
    return np.frombuffer(ctypes.string_at(address, 16 * N), dtype=complex)


class _Library:
    """Records the values behind the pointers of a call."""

    def __init__(self, places, status):
        self.places, self.status, self.seen = places, status, None

    def __getattr__(self, name):
        if name.startswith("dwf_mg_default"):
            return lambda p: None
        if name == "dwf_last_error":
            return lambda: b"stand-in"

        def call(*args):
            self.seen = [_values(args[i]).copy() for i in self.places]
            return self.status
        return call


def _run(monkeypatch, places, status, call):
    fake = _Library(places, status)
    monkeypatch.setattr(binding, "lib", lambda: fake)
    if status:
        with pytest.raises(binding.DwfError):
            call()
    else:
        call()
    return fake.seen


def test_dot(monkeypatch):
    (x, xv), (y, yv) = _strided(1), _strided(2)
    seen = _run(monkeypatch, (0, 1), 0, lambda: binding.dwf_dot(x, y, stream=0))
    assert np.array_equal(seen[0], xv) and np.array_equal(seen[1], yv)


def test_setup(monkeypatch):
    (u, uv), (v, vv) = _strided(3), _strided(4)
    geom = binding.make_geom((8, 8), 4)
    seen = _run(monkeypatch, (1, 5), 1, lambda: binding.mg_setup(geom, u, 1.0, 0.1, {}, v, stream=0))
    assert np.array_equal(seen[0], uv) and np.array_equal(seen[1], vv)


def test_add_level(monkeypatch):
    (u, uv), (v, vv) = _strided(5), _strided(6)
    mg = SimpleNamespace(ptr=None)
    seen = _run(monkeypatch, (2, 3), 1, lambda: binding.mg_add_level(mg, {}, u, v, stream=0))
    assert np.array_equal(seen[0], uv) and np.array_equal(seen[1], vv)
