"""The tile tuner on a handle whose clock is simulated: it times the library's own choice
beside the table and keeps it when it is the fastest; a cached choice is used as long as the
tile ids mean what they meant when it was written."""
import json
import os
import re
from types import SimpleNamespace

import pytest

torch = pytest.importorskip("torch")

from paper_2509_08971_gb300 import autotune  # noqa: E402


class Handle:
    """What tune uses of HardHydro, with a cost per tile."""

    shape, bc6, extent, dtype, scheme, gamma = (64, 64, 64), (0,) * 6, (1.0, 1.0, 1.0), "float32", 0, 1.4

    def __init__(self, cost, table):
        self.cost, self.table, self.tile, self.now, self.timed = cost, table, None, 0.0, set()
        clock = lambda: self.now  # noqa: E731

        class Event:
            def __init__(self, enable_timing=False):
                pass

            def record(self, stream):
                self.at = clock()

            def elapsed_time(self, other):
                return other.at - self.at

        cuda = SimpleNamespace(Event=Event, synchronize=lambda: None, current_stream=lambda: None)
        self.torch = SimpleNamespace(cuda=cuda, empty_like=lambda U: U)

    def cfl_dt(self, U, cfl):
        return 1e-3

    def tile_count(self):
        return len(self.table)

    def tile_info(self, tile):
        return self.table[tile] if tile >= 0 else (32, 16, 4, 512)

    def set_kernel(self, kernel, tile=-1):
        self.tile = tile

    def stage(self, stage, U0, U, dt, out=None):
        self.timed.add(self.tile)
        self.now += self.cost[self.tile]


TABLE = [(32, 8, 32, 256), (32, 16, 64, 512)]


@pytest.fixture(autouse=True)
def empty_memory(monkeypatch):
    monkeypatch.setattr(autotune, "_memory", {})
    monkeypatch.delenv("HARD_HYDRO_TUNE_CACHE", raising=False)


@pytest.mark.parametrize("cost,best", [({-1: 1.0, 0: 3.0, 1: 2.0}, -1), ({-1: 2.0, 0: 1.5, 1: 1.0}, 1),
                                       ({-1: 1.0, 0: 1.0, 1: 1.0}, -1)])
def test_the_librarys_choice_is_timed(cost, best):
    m = Handle(cost, TABLE)
    got = autotune.tune(m, object())
    assert m.timed == {-1, 0, 1} and got["tile"] == best == m.tile
    assert got["info"] == m.tile_info(best)
    assert got["ms"] == pytest.approx(cost)


def test_a_cache_of_other_tables_is_not_used(tmp_path):
    path = str(tmp_path / "tune.json")
    cost = {-1: 3.0, 0: 2.0, 1: 1.0}
    assert autotune.tune(Handle(cost, TABLE), object(), cache_path=path)["tile"] == 1
    autotune._memory.clear()
    again = Handle(cost, TABLE)
    got = autotune.tune(again, object(), cache_path=path)
    assert got["cached"] and got["tile"] == 1 and not again.timed
    autotune._memory.clear()
    other = Handle({-1: 3.0, 0: 1.0, 1: 2.0}, TABLE[::-1])
    got = autotune.tune(other, object(), cache_path=path)
    assert not got["cached"] and got["tile"] == 0 and len(json.load(open(path))) == 2


def test_batch_cache_of_other_tables_is_not_used(monkeypatch):
    B = SimpleNamespace(nx=[8], ny=[1], bcs=(0,), gammas=(1.4,), dtype="float32")
    key = autotune._batch_key(B)
    monkeypatch.setattr(autotune, "BATCH_TABLE", ("warps", 4, 2))
    assert autotune._batch_key(B) != key


def test_batch_table_is_the_librarys():
    here = os.path.dirname(os.path.abspath(autotune.__file__))
    text = open(os.path.join(here, "csrc", "launch.h")).read()
    warps = re.search(r"BATCH_WARPS\[\] = \{([^}]*)\}", text).group(1)
    assert autotune.BATCH_TABLE == ("warps", *(int(w) for w in warps.split(",")))
