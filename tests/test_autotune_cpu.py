"""What the autotuner times: the renderer whose launch parameters it chooses,
whatever the size of the view."""
import types

import pytest

torch = pytest.importorskip("torch")

from paper_2001_02620_gb300 import autotune
from paper_2001_02620_gb300 import inputs as I


class _Event:
    def __init__(self, **kw):
        pass

    def record(self):
        pass

    synchronize = record

    def elapsed_time(self, other):
        return 1.0


class _Scene:
    n_quads, n_instances, stats = 4096, 256, {"tlas_depth": 3, "max_blas_depth": 4}

    def __init__(self):
        self.seen = []

    def render(self, views, albedo, params, outs=None, tuning=None):
        self.seen.append(dict(tuning))

    def check(self):
        pass


@pytest.mark.parametrize("w,h,proxy", [(16, 8, 1 << 22), (64, 64, 1 << 10)])
def test_candidates_are_timed_on_the_wavefront_renderer(monkeypatch, w, h, proxy):
    """The default renderer of a small view is the single kernel, which reads
    neither occupancy nor batch."""
    monkeypatch.setattr(torch.cuda, "Event", _Event)
    monkeypatch.setattr(torch.cuda, "current_device", lambda: 0)
    monkeypatch.setattr(torch.cuda, "get_device_properties",
                        lambda d: types.SimpleNamespace(name="fake", multi_processor_count=152))
    scene = _Scene()
    view = I.View(eye=(0.0, 0.0, 1.0), look=(0.0, 0.0, 0.0), up=(0.0, 1.0, 0.0), vfov_deg=40.0, w=w, h=h, spp=1)
    space = {"occupancy": [32, 40], "batch": [1, 2]}
    best = autotune.tune(scene, view, torch.zeros(1, 3), I.Params(max_depth=2), space=space, reps=1, cache_path=None,
                         proxy_paths=proxy)
    assert scene.seen and all(t["mode"] == 2 for t in scene.seen)
    assert "mode" not in best  # a small frame rendered with the choice may still take the single kernel
    scene.seen.clear()
    autotune.tune(scene, view, torch.zeros(1, 3), I.Params(max_depth=2), space={"mode": [1]}, reps=1, cache_path=None)
    assert all(t["mode"] == 1 for t in scene.seen)  # unless the renderer is what is searched
