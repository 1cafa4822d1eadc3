"""Solves that the marching kernels take use no tile: the tuner leaves the tile shape alone, steps nothing and
keeps nothing, and a cached shape of an earlier tuning is not set either."""
import json
import math
import types

import pytest

torch = pytest.importorskip("torch")

from paper_2512_19847_gb300 import api, autotune, tableaux  # noqa: E402


class Marching:
    """A handle without solves on tiles; anything the tuner would do to it fails."""
    uses_tiles = False
    tile = 2
    _params = {0: types.SimpleNamespace(nx=512, ny=512, precision=api.FP32_DEV, space_scheme=2, s=3)}

    def set_tile(self, t):
        raise AssertionError("tile set")

    def step(self, n):
        raise AssertionError("stepped")


def test_tile_is_left_alone(tmp_path, monkeypatch):
    monkeypatch.setattr(torch.cuda, "get_device_name", lambda: "fake GPU")
    path = tmp_path / "c.json"
    path.write_text(json.dumps({autotune.signature(Marching()): {"tile": 4, "ms_per_step": {"4": 1.0}}}))
    before = path.read_text()
    assert autotune.tune(Marching(), path=str(path)) == {"tile": 2, "ms_per_step": {}, "cached": False}
    assert path.read_text() == before


def _params(n, prec):
    return api.default_params(n, n, eps=1e-3, dt=0.1 * 2 * math.pi / n, tau=0.05, mach=1e-2, tableau=tableaux.gsa2(), precision=prec)


@pytest.mark.gpu
def test_uses_tiles_follows_the_solves():
    assert api.Solver(_params(64, api.FP64)).uses_tiles and api.Solver(_params(512, api.FP64)).uses_tiles
    assert api.Solver(_params(64, api.FP32_DEV)).uses_tiles and not api.Solver(_params(512, api.FP32_DEV)).uses_tiles
    b = api.Batch(_params(512, api.FP32_DEV), 3)
    b.attach(0, _params(512, api.FP32_DEV))
    tile = b.tile
    assert not b.uses_tiles
    assert autotune.tune(b, path=None) == {"tile": tile, "ms_per_step": {}, "cached": False}
    b.attach(1, _params(8, api.FP32_DEV))      # too narrow to march: and no tuned shape refuses it
    assert b.uses_tiles
    b.step(1)
    b.sync_status()
    r = autotune.tune(b, steps=1, path=None)
    assert list(r["ms_per_step"]) == ["3"] and r["tile"] == b.tile == 3
