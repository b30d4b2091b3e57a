"""The real-plan cache holds the plans of rfft3d, irfft3d and hartree_energy at two
sizes at once: calls that alternate between them create no plan twice.  CPU only, with
a stand-in for the plan class."""
import contextlib

from paper_2006_08435_gb300 import fft


class _Plan:
    made = []

    def __init__(self, *key):
        _Plan.made.append(key)

    @classmethod
    def fixed(cls, n, batch):
        return cls("fixed", n, batch)


def test_two_sizes_fit(monkeypatch):
    monkeypatch.setattr(fft, "RealPlan", _Plan)
    monkeypatch.setattr(fft.torch.cuda, "device", lambda dev: contextlib.nullcontext())
    for cache in ("_real_cache", "_fixed_cache"):
        monkeypatch.setattr(fft, cache, fft.collections.OrderedDict(), raising=False)
    _Plan.made.clear()
    for _ in range(3):
        for n in (48, 96):
            fft._get_real_plan(n, 8, "fp32", False, "none", 0, 0)
            fft._get_real_plan(n, 8, "fp32", True, "by_n", 0, 0)
            fft._get_real_plan(n, 8, "fp32", False, "none", 0, 0, fixed=True)
    assert len(_Plan.made) == 6


def test_fixed_plans_are_bounded(monkeypatch):
    monkeypatch.setattr(fft, "RealPlan", _Plan)
    monkeypatch.setattr(fft.torch.cuda, "device", lambda dev: contextlib.nullcontext())
    monkeypatch.setattr(fft, "_fixed_cache", fft.collections.OrderedDict())
    for batch in range(1, 3 * fft._REAL_CACHE_MAX):
        fft._get_real_plan(48, batch, "fp32", False, "none", 0, 0, fixed=True)
    assert len(fft._fixed_cache) == fft._REAL_CACHE_MAX
