"""The tuner's cache: an entry is used for the same device, cavity (or
ensemble) and library sources only."""
import json

import pytest

from paper_1604_03478_gb300 import autotune


class Cav:
    shape, face, precision, node_pairs, solid = (64, 64, 64), 0, 0, -1, 0
    grid = type("G", (), {"precision": 0})

    def __init__(self, **kw):
        self.__dict__.update(kw)
        self.tried = []

    def set_launch(self, bx, by):
        self.tried.append((bx, by))

    def step(self, n):
        pass

    sync = None


class Ens:
    n, precision, dims = 2, 0, [(20, 20, 20, 0), (30, 30, 30, 1)]

    def __init__(self, **kw):
        self.__dict__.update(kw)
        self.tried = []

    def set_launch(self, block, k, graph_steps):
        self.tried.append((block, k))

    def info(self):
        return dict(nodes=sum(a * b * c for a, b, c, _ in self.dims))

    def member(self, i):  # a view of a member, which has no grid of its own
        return object()

    step = sync = None


@pytest.fixture
def tuner(tmp_path, monkeypatch):
    import torch
    monkeypatch.setattr(autotune, "CACHE", str(tmp_path / "tune.json"))
    monkeypatch.setattr(autotune, "_device_key", lambda: "GPU")
    monkeypatch.setattr(autotune, "_time", lambda *a: 1.0)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda: None)
    return autotune


def test_an_entry_of_other_sources_is_not_used(tuner, monkeypatch):
    with open(tuner.CACHE, "w") as fh:  # as written before entries named the sources
        json.dump({"cavity|GPU|64x64x64|p0": {"shape": [32, 4]}, "ensemble|GPU|n2|35000|p0": {"shape": [64, 2]}}, fh)
    c, e = Cav(), Ens()
    tuner.tune_cavity(c)
    tuner.tune_ensemble(e)
    assert c.tried[:-1] == list(tuner.CAVITY_SHAPES) and e.tried[:-1] == list(tuner.ENSEMBLE_SHAPES)
    again = Cav()
    tuner.tune_cavity(again)
    assert len(again.tried) == 1  # the entry just written
    monkeypatch.setattr(tuner, "_code_key", lambda: "other")
    other = Cav()
    tuner.tune_cavity(other)
    assert other.tried[:-1] == list(tuner.CAVITY_SHAPES)


@pytest.mark.parametrize("differ", [dict(shape=(64, 64, 32)), dict(face=1), dict(precision=1),
                                    dict(node_pairs=0), dict(solid=1)])
def test_a_cavity_that_differs_is_measured(tuner, differ):
    tuner.tune_cavity(Cav())
    c = Cav(**differ)
    tuner.tune_cavity(c)
    assert c.tried[:-1] == list(tuner.CAVITY_SHAPES)


@pytest.mark.parametrize("differ", [dict(precision=1), dict(dims=[(20, 20, 20, 1), (30, 30, 30, 1)])])
def test_an_ensemble_that_differs_is_measured(tuner, differ):
    tuner.tune_ensemble(Ens())
    e = Ens(**differ)
    tuner.tune_ensemble(e)
    assert e.tried[:-1] == list(tuner.ENSEMBLE_SHAPES)
