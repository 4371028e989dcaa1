"""The tuner against the library's own heights: measured, kept unless clearly beaten, and restored by set_tile."""
import types

import pytest

from test_autotune import FakeBatch, autotune   # noqa: F401 (fixture)
from test_host_runtime import fake, library, run, simulation   # noqa: F401 (fixture)


class FakeSim:
    def __init__(self, nx=2000, ny=2000, storage=0, s_form=0):
        self.nx, self.ny, self.params = nx, ny, types.SimpleNamespace(storage=storage, s_form=s_form, f_form=0)
        self.tile, self.measured = None, []

    def set_stream(self, s):
        pass

    def set_tile(self, t, r):
        self.tile = (t, r)
        self.measured.append(r)

    def step(self, n):
        pass


def test_own_choice_is_kept_unless_clearly_beaten(autotune, monkeypatch):   # noqa: F811
    for other, want in ((0.995, (128, 0)), (0.98, (128, 48))):
        times = {(t, r): 2.0 for t in autotune.BATCH_THREADS for r in autotune.BATCH_ROWS}
        times[(128, 48)], times[(128, autotune.AUTO)] = other, 1.0
        b = FakeBatch()
        monkeypatch.setattr(autotune, "_time", lambda fn, reps, stream: times[b.tile])
        assert autotune.tune_batch(b)[:2] == want
        assert b.tile == (128, want[1] or autotune.AUTO)


def test_each_height_is_measured_once_and_the_cache_keeps_choices_not_numbers(autotune, monkeypatch):   # noqa: F811
    sims = [FakeSim()]
    monkeypatch.setattr(autotune, "_time", lambda fn, reps, stream: 1.0 if sims[-1].tile[1] == autotune.AUTO else 1.5)
    assert autotune.tune_sim(sims[0], reps=1)[:2] == (autotune.THREADS[0], 0)
    heights = sims[0].measured[:-1]
    assert len(set(heights)) == len(heights) and autotune.AUTO in heights and sims[0].tile[1] == autotune.AUTO
    # 9 strips, 304 and 152 CTAs in a wave: 61 and 125 rows
    assert 61 in heights and 125 in heights
    sims.append(FakeSim(1500, 1100))                   # another grid of the class: its own choice, not a height
    assert autotune.tune_sim(sims[1])[:2] == (autotune.THREADS[0], 0)
    assert sims[1].measured == [autotune.AUTO]
    sims.append(FakeSim(s_form=1))                     # other strips: measured
    autotune.tune_sim(sims[2], reps=1)
    assert len(sims[2].measured) > 5
    sims.append(FakeSim(300, 20))                      # heights beyond the grid are one
    autotune.tune_sim(sims[3], reps=1)
    assert sum(r != autotune.AUTO and r >= 20 for r in sims[3].measured) == 1


def set_tile_and_back():
    lbm, f, events = library()

    def ctas(act):
        f.fake_clear()
        act()
        return [(e.what, e.n) for e in events() if e.what in (b"k_march", b"k_batch")]

    s = simulation(lbm, 500, 400)
    s.set_kernel(lbm.LBM_KERNEL_ROWS)
    fresh = ctas(lambda: s.step(1))
    s.set_tile(0, 7)
    assert ctas(lambda: s.step(1)) != fresh
    s.set_tile(128, lbm.AUTO_ROWS)
    assert ctas(lambda: s.step(1)) == fresh
    batch = lbm.Batch()
    members = [simulation(lbm, 200 + 10 * i, 300) for i in range(5)]
    for m in members:
        batch.add(m)
    fresh = ctas(lambda: batch.step(1))
    assert len(fresh) == 1
    batch.set_tile(0, 97)
    assert ctas(lambda: batch.step(1)) != fresh
    batch.set_tile(0, 0)
    assert ctas(lambda: batch.step(1)) != fresh        # 0 keeps
    batch.set_tile(0, lbm.AUTO_ROWS)
    assert ctas(lambda: batch.step(1)) == fresh


def test_auto_rows_restore_the_library_heights(fake):   # noqa: F811
    run(fake, "set_tile_and_back", module="test_autotune_own_choice")
