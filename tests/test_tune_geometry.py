"""The tuner against the library's present geometry: no two candidates are the
same cut, tiles of other kernels are not read from the cache, and a large batch
is not given tiles that are slower there than the automatic ones.  Host only."""
import json

import pytest
import torch

from paper_2203_02300_gb300 import tune
from paper_2203_02300_gb300.binding import Tile


@pytest.mark.parametrize("L1", [1, 34, 40])
def test_first_pass_candidates_are_different_cuts(L1):
    for n in (97, 320, 640, 641, 720, 1080, 1280, 1920, 4000):
        rows = set()
        for want in tune.first_pass_candidates(n, L1):   # k_hagg's ranges, by the rule of the library
            most = 640 - 2 * L1
            if n <= 640 and want == 0:
                cut = (n,)
            elif want == 0:
                cut = (640 - L1, most)
            else:
                assert want <= most, (n, want)
                cut = (-(-n // -(-n // want)),)
            assert cut not in rows, (n, want)
            rows.add(cut)
        cols = tune.first_pass_candidates(n, L1, 1)      # k_vcost's chunks
        assert all(c + 2 * L1 <= 1024 for c in cols[1:]) and len(set(cols)) == len(cols)
        assert n <= 1024 or 512 not in cols[1:]          # (512 is the automatic chunk)


def test_tiles_of_other_kernels_are_not_read(tmp_path, monkeypatch):
    path = tmp_path / "tiles.json"
    monkeypatch.setenv("DCO_TUNE_CACHE", str(path))
    path.write_text(json.dumps({"GPU|640x480|D64|o0|L34": {"tile": [32, 320, 96], "ms": {}}}))
    assert tune.lookup(640, 480, 64, "GPU") is None


@pytest.mark.parametrize("n,tuned_ms,want_tuned", [(32, 11.2, False), (32, 10.9, True), (2, 11.2, True)])
def test_a_large_batch_keeps_the_faster_tiles(tmp_path, monkeypatch, n, tuned_ms, want_tuned):
    monkeypatch.setenv("DCO_TUNE_CACHE", str(tmp_path / "tiles.json"))
    monkeypatch.setattr(torch.cuda, "get_device_name", lambda *a, **k: "fake GPU")
    shapes = [(1280, 720, 128)] * n
    won, timed = Tile(128, 0, 0), []

    class FakeStereo:
        def match_batch(self, pairs, params):
            timed.append([p[4] for p in pairs])

    def fake_time(fn, reps):
        fn()
        return 11.0 if timed[-1][0] == Tile() else tuned_ms
    monkeypatch.setattr(tune, "tune_shape", lambda *a, **k: won)
    monkeypatch.setattr(tune, "_time_call", fake_time)
    monkeypatch.setattr(tune, "_scene", lambda *a: (None, None), raising=False)
    monkeypatch.setattr(torch, "empty", lambda *a, **k: None)
    for _ in range(2):   # the second answer comes from the cache
        assert tune.tune_batch(FakeStereo(), shapes) == [won if want_tuned else Tile()] * n
    assert len(timed) == (2 if n == 32 else 0)
