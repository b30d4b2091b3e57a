"""The short path of fft3d(): the cases in which it must leave the fast accessors
aside, with stand-ins for the plan, the accessors and the tensor check (CPU only)."""
import contextlib

import pytest
import torch

from paper_2006_08435_gb300 import fft


class _Plan:
    def execute(self, x, out, stream):
        return ("plan", stream)


@pytest.fixture
def stand_ins(monkeypatch):
    switched = []
    monkeypatch.setattr(fft, "_check_tensor", lambda t, name: None)
    monkeypatch.setattr(fft, "get_plan", lambda *a: _Plan())
    monkeypatch.setattr(fft, "_current_stream_handle", lambda dev=None: 7)
    monkeypatch.setattr(fft, "_on_device",
                        lambda dev: switched.append(dev) or contextlib.nullcontext())
    monkeypatch.setattr(fft, "_plan_cache", {})
    return switched


@pytest.mark.parametrize("raw,current", [(None, None), (None, lambda: -1), (lambda d: 7, None),
                                         (lambda d: 7, lambda: 3)])
def test_a_missing_accessor_or_another_device_switches(stand_ins, monkeypatch, raw, current):
    monkeypatch.setattr(fft, "_raw_stream", raw)
    monkeypatch.setattr(fft, "_current_device", current)
    x = torch.zeros(4, 4, 4, dtype=torch.complex64)
    assert fft.fft3d(x) == ("plan", 7)
    assert stand_ins == [x.get_device()]


def test_no_grids_leave_out_unchecked(monkeypatch):
    """An empty batch returns `out` as it is."""
    seen = []
    monkeypatch.setattr(fft, "_check_tensor", lambda t, name: seen.append(name))
    x, out = torch.zeros(0, 4, 4, 4, dtype=torch.complex64), torch.zeros(3)
    assert fft.fft3d(x, out=out) is out
    assert seen == ["x"]
