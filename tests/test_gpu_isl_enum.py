"""ISL of rows from bit vectors at the edges of its words and kernels (one warp per row up
to L = 511, one CTA per row above), and the exhaustive search at the lengths where its
threads take one, a few and eight assignments at a time."""
from __future__ import annotations

import numpy as np
import pytest
import torch

import labs_inputs
import oracle
import paper_2011_00068_gb300 as labs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L", [3, 5, 31, 33, 63, 65, 95, 97, 127, 129, 255, 257, 479, 481, 511, 513, 545, 1023, 1025, 4097])
def test_isl_word_edges(L):
    B = 37 if L < 1000 else 5
    rows = labs_inputs.random_pm1((B, L), seed=L)
    rows[0] = 1
    rows[1] = labs_inputs.structured_pm1("alternating", L)
    rows[2, L - 1] = 0  # not +-1: ISL -1
    got = labs.isl(torch.from_numpy(rows).cuda()).cpu().numpy()
    want = [oracle.isl(np.ascontiguousarray(r)) for r in rows]
    want[2] = -1
    want = [-2 if w > 2 ** 31 - 1 else w for w in want]
    assert list(got) == [int(w) for w in want]


def test_isl_many_rows():
    """More rows than warps resident at once: every warp runs several."""
    L, B = 101, 40_001
    rows = labs_inputs.random_pm1((B, L), seed=3)
    got = labs.isl(torch.from_numpy(rows).cuda()).cpu().numpy()
    f = np.fft.rfft(rows.astype(np.float64), 256, axis=1)
    C = np.rint(np.fft.irfft(f * f.conj(), axis=1)[:, 1:L])
    assert np.array_equal(got, (C * C).sum(axis=1).astype(np.int64))


@pytest.mark.parametrize("L", [29, 33, 35, 37, 39, 41, 43])
def test_enumerate_matches_direct_search(L):
    """All assignments by numpy up to L = 33; above, the returned assignment reaches the
    minimum and no lower one does (up to 2^16 of them)."""
    c = (L - 1) // 2
    least, count, first = labs.enumerate_skew(L)
    a = np.arange(2 ** min(c, 16), dtype=np.int64)
    x = np.ones((a.size, c + 1), dtype=np.int8)
    x[:, :c] = 1 - 2 * ((a[:, None] >> np.arange(c)) & 1)
    j = np.arange(1, c + 1)
    rows = np.concatenate([x, x[:, c - j] * np.where(j % 2 == 1, -1, 1)], axis=1).astype(np.float64)
    f = np.fft.rfft(rows, 128, axis=1)
    C = np.rint(np.fft.irfft(f * f.conj(), axis=1)[:, 1:L])
    v = (C * C).sum(axis=1).astype(np.int64)
    if c <= 16:
        assert (least, count, first) == (v.min(), (v == v.min()).sum(), np.argmin(v))
    else:
        below = v[:min(first, v.size)]
        assert not (below <= least).any()
        xf = np.array([-1 if (first >> i) & 1 else 1 for i in range(c)] + [1], np.int8)
        assert oracle.isl(oracle.skew_expand(xf, L)) == least and count >= 1
