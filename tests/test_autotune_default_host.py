"""The tuner and the polymer's default launch shape: it is timed like the fixed blocks and, where it is
the fastest, left in place; a cached choice belongs to the kernels it was timed with."""
import json

import paper_1312_2213_gb300 as m
from paper_1312_2213_gb300 import autotune


class _Context:
    system, L, q, p, window = m.POLYMER3D, 32, 0, 4096, (53.0, 176.7)

    def __init__(self):
        self.set = []

    def set_param(self, key, value):
        self.set.append((key, value))


def test_default_shape_is_a_candidate_and_kept(tmp_path, monkeypatch):
    monkeypatch.setenv("MUCA_TUNE_CACHE", str(tmp_path / "tune.json"))
    g = _Context()
    r = autotune.apply(g, timer=lambda b: {None: 1.0, 128: 2.0, 256: 1.2, 512: 1.5}[b])
    assert r["block"] is None and r["ms"] == 1.0 and g.set == []
    r = autotune.apply(_Context(), timer=lambda b: 1 / 0)  # from the cache, null and all
    assert r["block"] is None
    g = _Context()
    autotune.apply(g, timer=lambda b: {None: 1.0, 128: 2.0, 256: 0.8, 512: 1.5}[b], use_cache=False)
    assert g.set == [("block", 256)]


def test_cache_belongs_to_the_kernels(tmp_path, monkeypatch):
    path = tmp_path / "tune.json"
    monkeypatch.setenv("MUCA_TUNE_CACHE", str(path))
    # an entry of earlier kernels (no tag in its key)
    path.write_text(json.dumps({"3/32/0/4096/test": {"block": 512, "ms": 0.1, "timings": {}}}))
    tune = lambda: autotune.tune(m.POLYMER3D, 32, 0, 4096, timer=lambda b: 1.0 if b == 128 else 2.0)
    assert tune()["block"] == 128
    monkeypatch.setattr(autotune, "_kernels", lambda: "others")
    assert autotune.tune(m.POLYMER3D, 32, 0, 4096, timer=lambda b: 1.0 if b == 256 else 2.0)["block"] == 256
    assert len(json.loads(path.read_text())) == 3
