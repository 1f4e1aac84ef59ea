"""Shared-memory bounds of the plain walk's step (csrc/labs_step.cuh), on the CPU.

tests/layout/step_dump.cpp prints the layout for every lane-group width and every longest
length of a context; for the lengths such a context may hold and the lane block the
kernel then takes, the extreme index of every family of accesses must stay in its region,
and what the product and the update read outside a class must be in the zero part."""
from __future__ import annotations

import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
FIELDS = "h0 hc ks r8 g gneg gpos z zneg x xp b bvec words R".split()


@pytest.fixture(scope="module")
def dump(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("layout") / "step_dump")
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", os.path.join(ROOT, "include"), "-I",
                    os.path.join(ROOT, "paper_2011_00068_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "layout", "step_dump.cpp"), "-o", exe], check=True)
    lay, shape = {}, {}
    for line in subprocess.run([exe], check=True, capture_output=True, text=True).stdout.splitlines():
        f = line.split()
        v = list(map(int, f[1:]))
        if f[0] == "step":
            lay[(v[0], v[1], v[2])] = dict(zip(FIELDS, v[3:]))
        else:
            shape[(v[0], v[1])] = (v[2], v[3], v[4])
    return lay, shape


def conflict_free(R, tile):
    while 16 // min(R & -R, 16) < tile // 2:
        R += 1
    return R


def check(S, shape, psl, tile, nmax, n, lay):
    RMAX = S["R"]
    R = lay[(psl, tile, n)]["R"]
    if tile == 32:
        R = RMAX if R >= RMAX else (RMAX - 2 if RMAX > 2 else 1)
    else:
        if R < RMAX - 3:
            R = conflict_free(RMAX - 3, tile)
        R = min(R, RMAX)
    M, NB, nR = shape[(tile, R)]                              # nR: the length the product is unrolled for
    assert n <= nR
    c, half, outs, walkers = n - 1, tile // 2, (tile // 2) * R, 32 // tile
    Sb, T, hw = (nR + 15) // 16, ((nR + 1) // 2 + 15) // 16, (n + 1) // 2
    lags = 4 * tile * NB                                      # lags the lanes' blocks cover
    assert T <= 4 * M and outs >= hw and lags >= n
    if n == nmax:
        assert lags >= S["gneg"] >= 16 * T
    pad1 = 2 * S["h0"] if psl else 8                          # copy 1's zero halves below its first word
    hlo, hhi = -2 * S["h0"], 2 * S["ks"] - pad1               # copy 0 of a class, halves
    klo, khi = -pad1, 2 * (S["hc"] - S["h0"] - S["ks"])      # copy 1, halves from its first word

    def row(u):
        assert hlo <= u < hhi, ("row", u)

    # entries written: copy 0 at u, copy 1 at u - 1
    for u in (0, n - 1):
        row(u)
        assert klo <= u - 1 < khi
    # s_{3i-L+1} of lanes with outputs; a class ends at n_p - 1
    for p in (0, 1):
        for lane in range(half):
            v0 = lane * R
            if 2 * v0 + p <= c:
                row(3 * v0 + p - n + 1)
                row(3 * v0 + p - n + 1 + 3 * (R - 1))
                zi = c - p - 2 * v0
            else:
                row(3 * (R - 1))
                zi = -1
            # Z: outputs that do not exist read the infinite part, the others m >= 0
            for r in range(R):
                m = zi - 2 * r
                assert -S["zneg"] <= m < lags
                assert (m < 0) == (not 2 * (v0 + r) + p <= c)
    if psl:  # pairs at v0 +- m, m = 1 .. n, in the copy of their parity; the list of lags
        for u in (-n, outs - R + n + R + 1):
            row(u - 1)
            row(u)
            assert klo <= u - 2 and u + 1 < khi
        assert S["x"] + n + 1 <= S["words"]
    # row blocks of the product: first diagonal -(T-1), last S-1 (with one operand, the load
    # of a last diagonal without a partner reads the next one's too)
    dlast = Sb - 1
    if walkers * M == 1 and (Sb + T - 1) % 2:
        dlast += 1
    tlast = 4 * M - 1
    row(16 * (-(T - 1)))
    row(16 * (tlast + dlast) + 15)
    # 16-byte operand rows
    assert S["h0"] % 4 == 0 and S["hc"] % 8 == 4 and S["words"] % 4 == 0
    # table words read by the product
    lo, hi = -7 - 16 * (T - 1) - 8, 6 + 16 * (Sb - 1) + 8
    assert -S["gneg"] <= lo and hi < S["gpos"] and n <= S["gpos"]
    assert S["g"] + S["gpos"] <= S["z"] - S["zneg"] // 2 and S["g"] - S["gneg"] >= S["r8"] + S["xp"] + outs
    # 16-byte stores of the table (mirror blocks 4 lags down), 8-byte stores of Z
    assert S["g"] % 4 == 0 and S["gneg"] % 4 == 0 and S["gpos"] % 4 == 0 and S["z"] % 2 == 0 and S["zneg"] % 8 == 0
    # update: two words from min((v >> 1) + 2 lb, hw) in either copy
    assert 2 * (hw + 2) <= hhi and 2 * (hw + 2) <= khi
    # Z words, the results, the bit vectors
    assert S["z"] + lags // 2 <= S["x"]
    tb = min((outs + 15) // 16, 4 * M)
    assert tb >= T and 16 * tb <= S["xp"] and outs <= S["xp"]
    assert S["x"] + S["xp"] + max(16 * tb, outs) <= S["words"]
    assert (n - 1) // 32 + 1 < S["bvec"] and S["b"] + 2 * S["bvec"] <= S["words"]


@pytest.mark.parametrize("psl,tile", [(0, 8), (0, 16), (0, 32), (1, 16), (1, 32)])
def test_step_accesses_stay_in_their_regions(dump, psl, tile):
    lay, shape = dump
    for (q, t, nmax), S in lay.items():
        if (q, t) != (psl, tile):
            continue
        for n in sorted(set(range(2, nmax + 1, 5)) | {2, 3, 4, 5, nmax - 1, nmax} | set(range(max(2, nmax - 40), nmax + 1))):
            if 2 <= n <= nmax:
                check(S, shape, psl, tile, nmax, n, lay)
