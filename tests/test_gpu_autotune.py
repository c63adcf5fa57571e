"""The tile autotuner keeps the fastest tile, the one the batch already has
among them: boxes of a few cells default to chunks of a few planes, which
take a fraction of the time of any length of 16 or more."""
import time

import pytest

from paper_2606_12753_gb300 import inputs as I
from paper_2606_12753_gb300 import mhd

pytestmark = pytest.mark.gpu


def _ms(b, steps=20):
    b.step(1e-6, steps)
    best = 1e9
    for _ in range(5):
        t = time.perf_counter()
        b.step(1e-6, steps)
        best = min(best, time.perf_counter() - t)
    return best / steps * 1e3


def test_autotuning_does_not_lose_the_default(tmp_path):
    boxes = [I.random_state(d, seed=i, bc=(1, 1, 1)) for i, d in enumerate([(32, 30, 96), (40, 24, 80)])]
    b = mhd.Batch(boxes, "fp32")
    for i, q in enumerate(boxes):
        b.set_state(i, q.cell, q.face)
    default = b.tile()[0]
    assert default[2] < 16
    before = _ms(b)
    b.set_tile(*default[:2], 16)
    assert _ms(b) > 1.25 * before       # no fixed length comes near
    b.set_tile(*default)
    cache = str(tmp_path / "tiles.jsonl")
    tile, ms = b.autotune(trial_steps=100, cache_path=cache)
    assert _ms(b) <= 1.1 * before, (default, tile, ms, before)
    # a tile that nothing proposes is among the trials when the batch has it, and the cache names the winner
    assert b.autotune(trial_steps=1, cache_path=cache)[0] == tile
    b.close()


def test_cache_lines_of_fewer_lengths_are_not_applied(tmp_path):
    """A line that was tuned without the short lengths has another key."""
    box = I.random_state((24, 16, 64), seed=2)
    b = mhd.Batch([box], "fp32")
    b.set_state(0, box.cell, box.face)
    cache = tmp_path / "tiles.jsonl"
    b.autotune(trial_steps=1, cache_path=str(cache))
    line = cache.read_text()
    old = line.replace("|z2", "")
    assert old != line
    cache.write_text(old.replace(line[line.index('"tile"'):line.index(', "ms_')], '"tile": [8, 8, 128]'))
    tile, _ = b.autotune(trial_steps=1, cache_path=str(cache))
    assert tile != (8, 8, 128) and len(cache.read_text().splitlines()) == 2
    b.close()
