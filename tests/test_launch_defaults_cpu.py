"""Scene.set_launch(kind) asks for the defaults of a new scene: zero in every field, as the header says."""
import inspect
import re

from conftest import ROOT


def test_set_launch_defaults_are_the_headers(monkeypatch):
    from paper_2510_25660_gb300 import api
    calls = []
    monkeypatch.setattr(api, "mt_set_launch", lambda *a: calls.append(a))
    s = object.__new__(api.Scene)
    s.h = None
    s.set_launch(api.MT_LAUNCH_RENDER)
    assert calls == [(None, api.MT_LAUNCH_RENDER, 0, 0, 0, 0, 0)]
    text = re.sub(r"\s*\n \*\s*", " ", open(f"{ROOT}/include/mt_api.h").read())
    assert "all zeros restore the configuration of a new scene" in text
    assert "0 = none (the default of every kind)" in text


def test_a_plan_without_a_privatisation_depth_gets_the_default(monkeypatch, tmp_path):
    from paper_2510_25660_gb300 import api, autotune
    monkeypatch.setattr(autotune, "_key", lambda *a: "k")
    monkeypatch.setattr(autotune, "_load", lambda: {"k": dict(threads=128, tile=2, ctas_per_sm=0)})
    calls = []

    class Fake:
        def set_launch(self, *a):
            calls.append(a)
    autotune.apply(Fake(), "nlos", None, None, 1, 0)
    default = inspect.signature(api.Scene.set_launch).parameters["priv_bins"].default
    assert calls == [(api.MT_LAUNCH_NLOS, 128, 2, 0, default, 0)]
