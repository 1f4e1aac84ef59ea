"""The row kernels (csrc/labs_rows.cu) at their edges: a wrong byte in any 16-byte piece of
one row of a pair leaves its neighbour alone, odd batches, and, on the CPU, the extreme
index of what the kernel writes beside the step's own accesses (test_step_layout)."""
from __future__ import annotations

import numpy as np
import pytest

import labs_inputs
import oracle
from test_step_layout import dump  # noqa: F401  (the layouts fixture)


@pytest.mark.gpu
@pytest.mark.parametrize("L", [31, 33, 63, 127, 193, 255, 257, 319, 321, 385, 447, 511])
def test_wrong_bytes_stay_in_their_row(L):
    import torch
    import paper_2011_00068_gb300 as labs
    places = sorted({0, 15, 16, 17, L // 2 - 1, L // 2 + 1, L - 17, L - 16, L - 2, L - 1} & set(range(L)))
    xs = labs_inputs.random_free_vars(4, L, seed=L)
    good = [oracle.skew_expand(x, L) for x in xs]
    want = [oracle.neighbor_delta(r) for r in good]
    c = (L - 1) // 2
    rows, ok = [], []
    for k, j in enumerate(places):
        for v in (0, 3, -128, -2, 127, None):  # None: the sign changes, which breaks Eq. 4
            bad = good[k % 4].copy()
            bad[j] = -bad[j] if v is None else v
            if v is None and j == c:  # the centre flips alone: still a skew-symmetric row
                want.append(oracle.neighbor_delta(bad))
            kb = len(want) - 1 if v is None and j == c else -1
            # the wrong row first or second of its pair
            rows += [bad, good[(k + 1) % 4]] if k % 2 else [good[(k + 1) % 4], bad]
            ok += [kb, (k + 1) % 4] if k % 2 else [(k + 1) % 4, kb]
    rows.append(good[2])
    ok.append(2)
    got = labs.neighbor_delta(torch.from_numpy(np.stack(rows)).cuda()).cpu().numpy()
    for b, k in enumerate(ok):
        if k < 0:
            assert (got[b] == -2**31).all(), b
        else:
            assert np.array_equal(got[b], want[k]), b


def test_row_kernel_bounds(dump):  # noqa: F811
    lay, _ = dump
    for n in range(2, 257):
        tile = 16 if n <= 160 else 32
        S = lay[(0, tile, n)]
        R, NW, c, half = S["R"], (n + 31) // 32, n - 1, tile // 2
        # the byte pieces' entries in copy 0 of a class: halves 0 .. 32 NW - 1, aligned stores
        assert S["h0"] % 4 == 0 and S["hc"] % 4 == 0 and S["words"] % 4 == 0
        assert 32 * NW <= 2 * S["ks"] - 8
        # bit vectors (bytes 4 NW) and the outputs' sign words, inside the results' words
        assert NW <= S["bvec"] and S["b"] + 2 * S["bvec"] <= S["words"]
        assert ((half - 1) * R >> 5) + 1 < S["bvec"]
        # every lag's pair, its mirror down to gneg, and Z
        assert n - 1 < S["gpos"] and n - 1 < 2 * (S["x"] - S["z"])
        # results of every lane output, existing or not, below the table
        assert S["r8"] + tile * R <= S["g"] - S["gneg"] and n <= tile * R
        # Z and s_{3i-L+1} of the last lane output: read in StepLane's ranges
        assert max(c, -1) < 2 * (S["x"] - S["z"]) and 2 * R <= S["zneg"]
        # half the pairs of a lag in the words that are counted, unmasked ones below it
        for q in range(NW):
            for m in {max(1, 32 * q), min(32 * q + 31, n - 1)}:
                if not 32 * q <= m <= 32 * q + 31:
                    continue
                for np_ in (n, n - 1):
                    h = max(np_ - m, 0) // 2
                    words = (NW - q + 1) // 2
                    assert h <= 32 * words
                    for k in range(words):
                        if 32 * (k + 1) <= 16 * (NW - q - 2):
                            assert 32 * (k + 1) <= h
