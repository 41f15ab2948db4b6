"""Niti.copy_tensors hands raw pointers to the library only for tensors that match in shape, type and layout; anything else
raises or is copied by torch (CPU: the library is replaced by one that records calls)."""
import pytest
import torch


class _Library:
    def __init__(self):
        self.sizes = []

    def niti_copy_tensors(self, handle, stream, n, dst, src, sizes):
        self.sizes += list(sizes[:n])
        return 0


@pytest.fixture()
def niti(monkeypatch):
    from paper_2009_13108_b200 import Niti
    n = Niti.__new__(Niti)
    n.lib, n.h, n.device = _Library(), None, torch.device("cpu")
    monkeypatch.setattr(Niti, "_stream", lambda self: 0)
    return n


def test_mismatches_raise(niti):
    from paper_2009_13108_b200 import NitiError
    a = lambda *s: torch.zeros(s, dtype=torch.int8)  # noqa: E731
    for dsts, srcs in (([a(8), a(8)], [a(8)]), ([a(64)], [a(16)]), ([a(4, 4)], [a(16)])):
        with pytest.raises(NitiError):
            niti.copy_tensors(dsts, srcs)
    assert niti.lib.sizes == []


def test_strides_types_and_places_are_torchs(niti):
    src = torch.arange(-24, 24, dtype=torch.int8).view(6, 8)
    wide, turned, other = torch.zeros(6, 16, dtype=torch.int8), torch.zeros(8, 6, dtype=torch.int8), torch.zeros(6, 8, dtype=torch.int32)
    niti.copy_tensors([wide[:, ::2], turned.t(), other], [src, src, src])
    assert torch.equal(wide[:, ::2], src) and bool((wide[:, 1::2] == 0).all())
    assert torch.equal(turned.t(), src) and torch.equal(other, src.int())
    host = torch.zeros(6, 8, dtype=torch.int8)
    niti.copy_tensors([host], [src])                    # (not this object's GPU)
    assert torch.equal(host, src) and niti.lib.sizes == []
