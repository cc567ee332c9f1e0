"""The JSON cache of tuned launch shapes (host logic; the library calls are
replaced): a table is loaded only for the grid, options and kernels it was
measured with."""
import json
import types

import pytest

from paper_1306_0645_gb300 import build, fld, synth

torch = pytest.importorskip("torch")


@pytest.fixture
def tuner(monkeypatch):
    calls = []
    monkeypatch.setattr(torch.cuda, "get_device_name", lambda *a: "NVIDIA GB300")
    monkeypatch.setattr(fld, "fld_autotune", lambda ctx, reps=3: calls.append("tuned"))
    monkeypatch.setattr(fld, "fld_get_tuning", lambda ctx: [128, 608, 2])
    monkeypatch.setattr(fld, "fld_tuning_size", lambda ctx: 3)
    monkeypatch.setattr(fld, "fld_set_tuning", lambda ctx, table: calls.append(list(table)))
    return calls


def context(**over):
    return types.SimpleNamespace(_g=fld.make_grid(synth.Grid.cube(64)),
                                 params=fld.make_params(synth.Params(precision=synth.PREC_MIXED, **over)))


def test_cached_table_is_loaded_for_the_same_kernels_only(tuner, monkeypatch, tmp_path):
    path = str(tmp_path / "tune.json")
    # a table saved before the kernels had a version in its key
    with open(path, "w") as f:
        json.dump({"64x64x64_bc000_p1_NVIDIA_GB300": [256, 152, 8]}, f)
    assert fld.autotune(context(), path) == [128, 608, 2] and tuner == ["tuned"]
    assert fld.autotune(context(), path) == [128, 608, 2] and tuner[1:] == [[128, 608, 2]]
    # other kernels: measured again
    monkeypatch.setattr(build, "source_digest", lambda: "other")
    fld.autotune(context(), path)
    assert tuner[2:] == ["tuned"]


def test_cached_table_is_not_shared_between_sweep_options(tuner, tmp_path):
    path = str(tmp_path / "tune.json")
    for over in ({}, {"post": 2}, {"precond_bf16": 0}, {"tail_cells": 0}):
        fld.autotune(context(**over), path)
    assert tuner == ["tuned"] * 4
    fld.autotune(context(post=2), path)
    assert tuner[4:] == [[128, 608, 2]]
