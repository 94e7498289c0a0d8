"""The tuner and the default route: the route of a table whose shapes nobody has set is
a candidate like the others, and `apply()` does not take bulk calls away from a table
that is large enough for them."""
import json

import pytest

from paper_1908_05936_gb300 import _lib as L
from paper_1908_05936_gb300 import tune


class FakeTable:
    kind, bucket_bytes = L.MAP_U64_U64, 64

    def __init__(self, table_bytes):
        self.nb, self.set = table_bytes // self.bucket_bytes, {}

    def device_view(self):
        return self

    def set_launch(self, op, **shape):
        self.set[op] = shape


@pytest.fixture
def cache(tmp_path, monkeypatch):
    shape = dict(lane_bytes=32, keys_per_group=4, block=64, ms=1.0, mops=1.0)
    path = tmp_path / "tuned.json"
    path.write_text(json.dumps({"dev/1SM": {"map_u64_u64/64": {
        "insert": shape, "find": dict(default=True, ms=1.0, mops=1.0), "find_hit": shape, "find_miss": shape,
        "erase": shape}}}))
    monkeypatch.setattr(tune, "CACHE", str(path))
    monkeypatch.setattr(tune, "device_key", lambda: "dev/1SM")


def test_apply_installs_shapes_on_small_tables(cache):
    t = FakeTable(100 << 20)
    assert tune.apply(t)
    assert t.set == {op: dict(lane_bytes=32, keys_per_group=4, block=64) for op in (L.OP_INSERT, L.OP_ERASE)}


def test_apply_leaves_large_tables_their_bulk_calls(cache):
    t = FakeTable(512 << 20)
    assert tune.apply(t) and t.set == {}


def test_the_default_route_wins_unless_clearly_beaten():
    d, s = dict(default=True), dict(lane_bytes=32)
    assert tune.fastest([(1.0, d), (0.98, s)]) == (1.0, d)
    assert tune.fastest([(1.0, d), (1.2, dict(block=64)), (0.9, s)]) == (0.9, s)


@pytest.mark.gpu
@pytest.mark.parametrize("kind,bb", ((L.SET_U64, 32), (L.MAP_U64_U64, 64)))
def test_tune_table_times_the_default_route_first(kind, bb):
    rows = []
    best = tune.tune_table(kind, bb, slots_log2=16, every=rows)
    assert rows[0]["default"] and not any(r.get("default") for r in rows[1:])
    assert all(best[op].get("default") or best[op]["keys_per_group"] in (1, 2, 4, 8)
               for op in ("insert", "find", "find_hit", "find_miss", "erase"))
