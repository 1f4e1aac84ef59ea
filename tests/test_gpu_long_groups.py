"""Lengths on both sides of the line between the long product's two forms (n = 512) in one
context, on the same CTAs one after the other: each walker as in a context of its own length."""
from __future__ import annotations

import numpy as np
import pytest

import paper_2011_00068_gb300 as labs
from paper_2011_00068_gb300 import _native

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("flags", [0, _native.LABS_FLAG_BEST_FIRST, _native.LABS_FLAG_PSL])
@pytest.mark.parametrize("Ls", [(1023, 1025), (1025, 1023), (513, 1279)])
def test_two_forms_in_one_context(Ls, flags):
    W, steps = 700, 24  # more walkers than CTAs
    s = labs.Search(list(Ls), [W, 5], 9, tabu_log2=8, flags=flags, chunk_steps=8)
    s.walk(steps)
    s.sync()
    mixed = s.results(0, W)
    s.close()
    s = labs.Search(Ls[0], W, 9, tabu_log2=8, flags=flags, chunk_steps=8)
    s.walk(steps)
    s.sync()
    alone = s.results(0, W)
    s.close()
    for k in ("isl", "best_isl"):
        assert np.array_equal(mixed[k], alone[k]), k
