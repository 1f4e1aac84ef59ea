"""The long sequences' tensor-core product: the neighbourhood at the edges of its column
groups (two to four at once) and CTA widths, a table entry that FP16 does not hold, and, on
the CPU, the extreme table, row and result index of every set of groups."""
from __future__ import annotations

import numpy as np
import pytest

import labs_inputs
import oracle
from test_layout_bounds import Region, layouts  # noqa: F401  (the layouts fixture)


@pytest.mark.gpu
@pytest.mark.parametrize("n", [257, 272, 384, 385, 512, 513, 640, 641, 767, 769, 1025, 1152, 1153, 1665, 2304, 2305,
                               2561, 3649, 4608, 4609])
def test_long_neighbourhood_at_group_edges(n):
    import torch
    import paper_2011_00068_gb300 as labs
    L = 2 * n - 1
    rows = np.stack([oracle.skew_expand(x, L) for x in labs_inputs.random_free_vars(3, L, seed=n)])
    got = labs.neighbor_delta(torch.from_numpy(rows).cuda()).cpu().numpy()
    for k, r in enumerate(rows):
        assert np.array_equal(got[k], oracle.neighbor_delta(r)), k


@pytest.mark.gpu
def test_long_neighbourhood_with_an_autocorrelation_above_2048():
    """x symmetric about c - 2048 (with the signs of Eq. 4) makes every term of C_4096 a
    +1: C_4096 = L - 4096 = 4095, an odd number above 2^11, beside small ones."""
    import torch
    import paper_2011_00068_gb300 as labs
    L = 8191
    n = (L + 1) // 2
    x = labs_inputs.random_free_vars(1, L, seed=8)[0].copy()
    c = n - 1
    for a in range(4096 - c, 2048):
        x[c - (4096 - a)] = x[c - a] * (-1) ** a
    x = np.ascontiguousarray(x)
    row = oracle.skew_expand(x, L)
    assert int((row[:L - 4096].astype(np.int64) * row[4096:]).sum()) == 4095
    plain = oracle.skew_expand(labs_inputs.random_free_vars(1, L, seed=9)[0], L)
    rows = np.stack([plain, row, plain])
    got = labs.neighbor_delta(torch.from_numpy(rows).cuda()).cpu().numpy()
    for k, r in enumerate(rows):
        assert np.array_equal(got[k], oracle.neighbor_delta(r)), k


def test_long_product_bounds(layouts):  # noqa: F811
    bad = []
    for (nt, n_max), lay in layouts[1].items():
        if not lay["xp"]:
            continue
        assert lay["hlen"] % 8 == 4 and lay["hoff"] % 4 == 0 and lay["hpad"] % 8 == 0  # ldmatrix rows
        assert (lay["roff"] + 2 * lay["xp"]) % 4 == 0                                  # the mark follows
        assert lay["words"] >= lay["roff"] + 2 * lay["xp"] + 4
        for n in {257, (257 + n_max) // 2, n_max}:
            reg = Region(lay)
            S, T = (n + 15) >> 4, (((n + 1) >> 1) + 15) >> 4
            M, C = (T + 3) >> 2, (S - 1) >> 2
            Q = (M + 3) >> 2
            few, more, m0, total = M // Q, M % Q, 0, 0
            for q in range(Q):
                gc = few + (q < more)
                assert gc in (2, 3, 4)
                for k in (-(m0 + gc), C - m0):          # first and last chunk of the set
                    reg.g(64 * k - 7 - 8, "table")
                    reg.g(64 * k + 48 + 6 + 8 + 1, "table")
                    reg.h(64 * (k + m0), "rows")
                    reg.h(64 * (k + m0 + gc - 1) + 16 * (3 + 3) + 15, "rows")
                total += C + 1 + gc
                m0 += gc
            assert m0 == M and total == Q * (C + 1) + M and 16 * T <= lay["xp"]
            bad += [(nt, n_max, n, b) for b in reg.bad[:2]]
    assert not bad, bad[:5]
