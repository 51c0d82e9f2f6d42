"""The autotuner leaves alone what does not run the kernels it shapes (planning only, no GPU)."""
import dataclasses
import os

import pytest

import paper_2103_09686_gb300 as dm
from paper_2103_09686_gb300 import tune


@pytest.mark.parametrize("p", [
    dm.Params(shape=(512, 512), window=(64, 64), levels=3),                              # separable
    dm.Params(shape=(128, 128, 128), window=(24, 24, 24), levels=2),
    dm.Params(shape=(256, 256), window=(32, 32), levels=3, phases=2),
    dm.Params(shape=(256, 256), window=(64, 64), descriptor=dm.DMCR_DESC_S2_TILDE),
    dm.Params(shape=(64, 64, 64), window=(24, 24, 24), threshold=dm.DMCR_IDENTITY),      # FFT, by AUTO
    dm.Params(shape=(64, 64), window=(8, 8), threshold=dm.DMCR_IDENTITY, path=dm.DMCR_PATH_FFT),
])
def test_other_paths_are_not_tuned(tmp_path, monkeypatch, p):
    monkeypatch.setattr(tune, "search", lambda *a, **k: pytest.fail("measured"))
    monkeypatch.setattr(tune, "_key", lambda q: "key")
    cache = str(tmp_path / "tune.json")
    assert tune.tuned(p, cache) is p and not os.path.exists(cache)


@pytest.mark.parametrize("p", [dm.Params(shape=(64, 64), window=(16, 16), levels=2),
                               dm.Params(shape=(96, 64), window=(12, 9), levels=2),
                               dm.Params(shape=(512, 512), window=(64, 64), levels=3, path=dm.DMCR_PATH_DIRECT),
                               dm.Params(shape=(56, 56), window=(8, 8), threshold=dm.DMCR_IDENTITY),
                               # its finest level goes to the transforms, the others do not
                               dm.Params(shape=(128, 128, 128), window=(6, 6, 6), levels=3, threshold=dm.DMCR_IDENTITY)])
def test_direct_problems_are_tuned(tmp_path, monkeypatch, p):
    monkeypatch.setattr(tune, "search", lambda *a, **k: ((8, 2, 0, 3), 1.0, []))
    monkeypatch.setattr(tune, "_key", lambda q: "key")
    q = tune.tuned(p, str(tmp_path / "tune.json"))
    assert q == dataclasses.replace(p, tune=(8, 2, 0, 3))
