"""Stop requests are asked for at the steps where a walker's own count is a multiple of 64,
whatever the chunks (the question waits for host memory: at every chunk's start it took a
third of a one-step chunk)."""
from __future__ import annotations

import pytest

import paper_2011_00068_gb300 as labs
from paper_2011_00068_gb300 import _native

pytestmark = pytest.mark.gpu

EVERY = 64


@pytest.mark.parametrize("L,W,flags", [(41, 9, 0), (41, 700, 0), (201, 6, 0), (201, 200, 0), (401, 5, 0), (401, 90, 0),
                                       (201, 7, _native.LABS_FLAG_PSL), (303, 7, _native.LABS_FLAG_PSL),
                                       (101, 5, _native.LABS_FLAG_BEST_FIRST)])
@pytest.mark.parametrize("chunk", [1, 5])
def test_checks_come_every_64_steps(L, W, flags, chunk):
    s = labs.Search(L, W, 3, tabu_log2=10, chunk_steps=chunk, flags=flags)
    s.walk(10)
    s.sync()
    s.set_deadline(0)
    s.walk(20)  # no step of these is a multiple of 64
    s.sync()
    assert s.stats()["steps"] == 30 * W
    s.walk(EVERY)
    with pytest.raises(labs.LabsError) as err:
        s.sync()
    assert err.value.code == _native.LABS_ETIMEOUT
    s.clear_stop()
    assert s.stats()["steps"] == EVERY * W
    s.walk(0)
    s.sync()
    assert s.stats()["steps"] == (30 + EVERY) * W
    s.close()
