"""The tuner times what differs: one run of updates for each kernel that the accepted codes choose
between, every code's time reported, and never one of two codes of the same kernel picked by noise."""
import itertools
import types

import pytest

torch = pytest.importorskip("torch")

from paper_2511_16633_gb300 import rb, tune  # noqa: E402


class _Event:
    clock = itertools.count()

    def __init__(self, enable_timing=False):
        self.at = 0

    def record(self, stream=None):
        self.at = next(_Event.clock)

    def synchronize(self):
        pass

    def elapsed_time(self, other):
        return float(other.at - self.at) / (1 + next(_Event.clock))   # every reading another


@pytest.mark.parametrize("prec,single", [(rb.RB_PREC_FP32, 0), (rb.RB_PREC_BF16X3, rb.RB_TUNE_ADJ_SINGLE)])
def test_each_form_is_timed_once(monkeypatch, prec, single):
    calls = []
    null = types.SimpleNamespace(__enter__=lambda s: None, __exit__=lambda s, *a: None)
    monkeypatch.delenv("RB_TUNE_CACHE", raising=False)
    monkeypatch.setattr(tune, "_cache", {})
    monkeypatch.setattr(torch.cuda, "Stream", lambda device=None: None)
    monkeypatch.setattr(torch.cuda, "stream", lambda s: type("C", (), {"__enter__": null.__enter__, "__exit__": null.__exit__})())
    monkeypatch.setattr(torch.cuda, "Event", _Event)
    monkeypatch.setattr(rb, "workspace", lambda *a, **k: None)
    monkeypatch.setattr(rb, "rb_hf_update", lambda *a, **k: calls.append(k["tune"]))
    geom = rb.geometry(64, 0.05, 64, 64, 2e-3, 32)
    best, info = tune.tune_update(geom, torch.zeros(4), None, [1e6], torch.zeros(1), prec, reps=3)
    forms = [single | r for r in (rb.RB_TUNE_RASTER_ALONG, rb.RB_TUNE_RASTER_ACROSS)]
    assert sorted(set(calls)) == sorted(forms) and len(calls) == 2 * 4    # a warm-up and three runs of each
    assert best in forms
    assert set(info["ms_per_update"]) == {tune.name(t) for t in tune.candidates(prec)}
    for t in tune.candidates(prec):   # a code's time is that of the kernel it runs
        assert info["ms_per_update"][tune.name(t)] == info["ms_per_update"][tune.name(single | (t & 3))]
