"""The shape search reaches a tuned walk although the library's default, packets of
rays, beats every walk whose other fields are at their defaults, and returns the default
where no walk beats it (host logic, no GPU)."""
import pytest

from paper_2005_06671_gb300 import autotune

TARGET = {"block_threads": 128, "rays_per_thread": 64, "ray_tile_w": 32, "refill_min": 10,
          "leaf_level": 2, "strip_len": 0}


@pytest.mark.parametrize("packets,best", [(60.0, TARGET), (20.0, autotune.DEFAULT)])
def test_search_descends_over_the_walks(monkeypatch, packets, best):
    timed = []

    def fake_time(hfs, suns, lmax, p, reps, step):
        assert autotune._valid(p), p
        timed.append(tuple(sorted(p.items())))
        if p == autotune.DEFAULT:
            return packets
        return 50.0 + 20.0 * sum(abs(autotune.SPACE[k].index(p[k]) - autotune.SPACE[k].index(TARGET[k]))
                                 for k in p)

    monkeypatch.setattr(autotune, "time_batch", fake_time)
    got, seen = autotune.tune([], [], 50e3, reps=1, rounds=3)
    assert got == best
    assert len(timed) == len(set(timed)) == len(seen)
