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


@pytest.mark.parametrize("kind", ["list", "array", "subclass", "other"])
def test_evolve_takes_media_of_its_own_layout_only(kind):
    """An array of media is handed on as it is; one of a larger structure is converted as a list of media is, and one of
    another type is refused."""
    import ctypes as C
    from paper_2107_06147_gb300 import qtraj

    class Larger(qtraj.Medium):
        _fields_ = [("note", C.c_int)]

    got = []

    def evolve(ctx, batch, media, n_media, idx, seeds, stream):
        p = C.cast(media, C.POINTER(qtraj.Medium))
        got.append([p[i].T0 for i in range(n_media)])
        return 0

    e = object.__new__(qtraj.Engine)
    e.ctx, e.lib = None, types.SimpleNamespace(qtraj_evolve=evolve)
    m = [qtraj.medium(0.4 + 0.01 * i) for i in range(3)]
    if kind == "array":
        m = (qtraj.Medium * 3)(*m)
    elif kind == "subclass":
        m = (Larger * 3)(*[Larger(0, 0.4 + 0.01 * i, 0.6, 0.25, 5.0, 0.0, 0, 0, 1) for i in range(3)])
    elif kind == "other":
        with pytest.raises(TypeError):
            e.evolve((C.c_double * 3)(1.0, 2.0, 3.0), np.arange(3), stream=0)
        return
    e.evolve(m, np.arange(3), stream=0)
    assert np.allclose(got[0], [0.4, 0.41, 0.42])
