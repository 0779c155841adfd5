"""The launch-shape search times the library's automatic setting beside the requested shapes (no GPU: a stand-in context
and clock).  A requested shape turns the evaluation by unordered pairs off, so it is kept only where it is faster."""
import pytest


class FakeContext:
    precision = 1

    def __init__(self, n):
        self.n = n
        self.tiles = None
        self.lists = []

    def set_tiles(self, **shape):
        self.tiles = shape

    def resolve_tiles(self, n_act):
        return {}


class FakeList:
    def __init__(self, k):
        self.k = k

    def numel(self):
        return self.k


@pytest.mark.parametrize("automatic,n_act", [(0.5, 1000), (2.0, 1000), (0.5, 4096), (2.0, 4096)])
def test_automatic_setting_is_a_candidate(monkeypatch, tmp_path, automatic, n_act):
    autotune = pytest.importorskip("paper_1901_08532_gb300.autotune")
    monkeypatch.setattr(autotune, "_cache", {})
    fast = {"ki": 2, "junroll": 4, "threads": 128, "jtile": 512, "lanes": 2}

    def clock(ctx, shape, active, reps=3):
        ctx.set_tiles(**shape)
        ctx.lists.append(active)
        return automatic if not shape else 1.0 if shape == fast else 3.0

    monkeypatch.setattr(autotune, "time_shape", clock)
    ctx, active, cache = FakeContext(4096), FakeList(n_act), str(tmp_path / "shapes.json")
    want = ({}, 0.5) if automatic < 1.0 else (fast, 1.0)
    assert autotune.tune(ctx, active, cache_file=cache) == want
    assert ctx.tiles == want[0]
    # all particles are timed as such: only the implied list takes unordered pairs
    assert all(a is (None if n_act == ctx.n else active) for a in ctx.lists)
    # from the file, without timing
    monkeypatch.setattr(autotune, "_cache", {})
    again = FakeContext(4096)
    assert autotune.tune(again, active, cache_file=cache) == want
    assert again.tiles == want[0] and not again.lists
