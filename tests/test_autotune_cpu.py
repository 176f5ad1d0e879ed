"""The autotuner times each tile shape once: nothing else that it could vary has an
effect at its tiles, and the choice must not come from repeated noise."""
import json

import pytest

from paper_2409_13055_gb300 import autotune, mapping, scenes


class _Map:
    n = 1000


@pytest.fixture
def timed(monkeypatch, tmp_path):
    tiles = []

    def fake(views, gmap, targets, lam, tile, iters, tight_rect=True):
        tiles.append((tile, iters))
        return dict(zip(autotune.TILES, ((1.0, 0.3, 0.5), (0.9, 0.35, 0.4), (1.1, 0.2, 0.6))))[tile]

    monkeypatch.setattr(autotune, "_time_tile", fake, raising=False)
    # (what an earlier tuner called once per batch and pixels per thread)
    monkeypatch.setattr(autotune, "_time_config",
                        lambda v, g, t, lam, tile, batch, ppt, iters, tight=True:
                        fake(v, g, t, lam, tile, iters), raising=False)
    monkeypatch.setattr(autotune, "cache_key", lambda *a: "key")
    monkeypatch.setenv("GS_AUTOTUNE_CACHE", str(tmp_path / "tuned.json"))
    return tiles


def test_each_tile_is_timed_once_and_the_choice_is_one_that_was_timed(timed, tmp_path):
    got = autotune.autotune([], _Map, None, 0.2, iters=5)
    assert [t for t, _ in timed] == list(autotune.TILES)
    assert got["tile"] == (16, 16) and got["ms"] == 0.9 and len(got["timings"]) == 3
    again = autotune.autotune([], _Map, None, 0.2)
    assert again["cached"] and len(timed) == 3
    assert {k: v for k, v in again.items() if k not in ("cached", "timings")} == \
        {k: v for k, v in got.items() if k not in ("cached", "timings")}
    assert json.loads((tmp_path / "tuned.json").read_text())["key"]["tile"] == [16, 16]


@pytest.mark.parametrize("tile", autotune.TILES)
def test_the_shape_is_one_that_every_plan_of_the_tile_takes(timed, tile, monkeypatch):
    monkeypatch.setattr(autotune, "TILES", (tile,))
    got = autotune.autotune([], _Map, None, 0.2, use_cache=False)
    keys = ("smem_batch", "pixels_per_thread", "smem_batch_bwd", "pixels_per_thread_bwd")
    view = scenes.camera(64, 48, 50.0, 50.0)
    for det in (False, True):
        assert mapping.plan_workspace_bytes([view], 100, 1000, tile=tile, deterministic=det,
                                            **{k: got[k] for k in keys}) > 0
