"""Host logic of the tuner, with a solver and a batch that only record their calls: the timed solves of a
dt come after its capture (the first solve of a dt launches directly, the second captures), and the tile
mappings tried are distinct (their two numbers multiply)."""
import types

import numpy as np

from paper_1912_06221_gb300 import autotune, rdg

LOG = []


class Event:
    def __init__(self, enable_timing):
        pass

    def record(self, stream):
        LOG.append("record")

    def elapsed_time(self, other):
        return 1.0


TORCH = types.SimpleNamespace(cuda=types.SimpleNamespace(Event=Event, synchronize=lambda: None))


class Solver:
    stream, N = None, 3

    def set_state(self, u):
        pass

    def solve_to_time(self, t0, dt, n):
        LOG.append("solve")


class Batch:
    stream, mode = None, rdg.BATCH_PERSISTENT

    def __init__(self):
        self.tiles = []

    def set_tiles(self, N, e, tpi):
        self.tiles.append((N, e * tpi))

    def set_mode(self, m):
        pass

    def step(self, n):
        pass


def test_timed_solves_come_after_the_capture():
    del LOG[:]
    autotune._time_steps(TORCH, Solver(), np.zeros(1), 1e-3, 16)
    assert LOG[: LOG.index("record")].count("solve") >= 2


def test_tile_mappings_tried_are_distinct(monkeypatch):
    monkeypatch.setitem(__import__("sys").modules, "torch", TORCH)
    b = Batch()
    out = autotune.choose_tiles(b, [Solver()], [np.zeros(1)], 4)
    tried = b.tiles[:-1]                                  # the last call leaves the best
    assert len(tried) == len(set(tried)) and {t for _, t in tried} == {1, 2, 4, 8}
    assert b.tiles[-1] in tried and 3 in out["edges_per_thread_tiles_per_item"]
