"""The tiling search times each launch once: with a whole pair per lane the
tile and grid fields do not reach the library's launch."""
from paper_2103_14978_gb300 import batch


class Fake:
    def __init__(self, *args):
        self.tiling = args[-1]


def search(monkeypatch, ms):
    timed = []
    monkeypatch.setattr(batch, "BatchedFilter", Fake)
    monkeypatch.setattr(batch, "_time", lambda bf, reps: timed.append(bf.tiling) or ms(bf.tiling))
    best, results = batch.autotune(*[None] * 9)
    return best, timed, results


def test_one_pair_per_lane_is_one_candidate(monkeypatch):
    best, timed, results = search(monkeypatch, lambda t: 1.0 if t[0] == 1 else 2.0 + t[0])
    assert best == batch.DEFAULT_TILING
    assert [t[0] for t in timed].count(1) == 1
    assert len(timed) == len(results) == len(batch.WPT_CHOICES)


def test_lane_groups_search_tiles_and_grids(monkeypatch):
    best, timed, _ = search(monkeypatch, lambda t: (5.0 if t[0] == 1 else 1.0 + abs(t[0] - 4)) + (t[1] != 64) +
                            (t[2:] != (8, 4)))
    assert best == (4, 64, 8, 4)
    assert len(timed) == len(set(timed))
