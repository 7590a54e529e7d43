"""The uneven batch's host side: media that the caller changes between calls (CPU, with a stand-in for the engine)."""
import types

import numpy as np
import pytest


def test_media_changed_between_calls_take_effect(monkeypatch):
    torch = pytest.importorskip("torch")
    from paper_2107_06147_gb300 import batching, qtraj
    calls = []

    class Engine:
        def __init__(self, cfg):
            self.N = cfg.N

        def init(self, specs, n, spec_idx=None):
            pass

        def evolve(self, media, seeds, medium_idx=None, batch=None, stream=None):
            calls.append((self.N, [media[i].kappa_hat for i in medium_idx], list(seeds)))

    monkeypatch.setattr(qtraj, "Engine", Engine)
    monkeypatch.setattr(torch.cuda, "Stream", types.SimpleNamespace)
    media = [qtraj.medium(0.4, 0.6, 0.3 + 0.01 * i, float(i), 0.0) for i in range(5)]
    b = batching.UnevenBatch([32, 64, 32, 64, 32], [qtraj.init_spec()] * 5, media)
    for m in media:
        m.kappa_hat += 10.0
    b.evolve(np.arange(5))
    assert [c[0] for c in calls] == [64, 32]
    for _, kappa, seeds in calls:
        assert kappa == [10.0 + s for s in seeds]
    media[3].kappa_hat = 7.0
    calls.clear()
    b.evolve(np.arange(5))
    assert dict(zip(calls[0][2], calls[0][1]))[3] == 7.0
