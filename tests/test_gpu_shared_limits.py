"""Contexts, lengths and host threads that share a kernel and need different amounts of shared
memory: none takes away what another one's launch needs."""
from __future__ import annotations

import threading

import numpy as np
import pytest
import torch

import paper_2011_00068_gb300 as labs
from paper_2011_00068_gb300 import _native

pytestmark = pytest.mark.gpu


def skew(L, rows, seed):
    rng = np.random.default_rng(seed)
    x = (1 - 2 * rng.integers(0, 2, (rows, (L + 1) // 2))).astype(np.int8)
    j = np.arange(1, x.shape[1])
    s = np.concatenate([x, x[:, x.shape[1] - 1 - j] * np.where(j % 2 == 1, -1, 1).astype(np.int8)], axis=1)
    return np.ascontiguousarray(s.astype(np.int8))


# both lengths of a pair run the same kernels (lane block and threads), the second with less
@pytest.mark.parametrize("L,less,flags", [(1791, 1283, 0), (1791, 1283, _native.LABS_FLAG_BEST_FIRST),
                                          (1535, 601, _native.LABS_FLAG_PSL)])
def test_a_shorter_context_leaves_a_longer_one_its_memory(L, less, flags):
    W, steps = 3, 40
    a = labs.Search(L, W, 5, tabu_log2=10, flags=flags)
    b = labs.Search(less, W, 5, tabu_log2=10, flags=flags)
    a.reset()
    a.walk(steps)
    a.sync()
    b.walk(steps)
    b.sync()
    assert a.stats()["steps"] == W * steps and b.stats()["steps"] == W * steps
    a.close()
    b.close()


def test_row_kernels_from_several_threads():
    """Two lengths of one row kernel, many and few rows, each from a thread of its own on a
    stream of its own; every result as from one thread."""
    work = [(223, 4096), (193, 4096), (223, 700), (201, 64), (511, 3000), (387, 2000)]
    rows = [torch.from_numpy(skew(L, B, 7 + k)).cuda() for k, (L, B) in enumerate(work)]
    want = [labs.neighbor_delta(r).clone() for r in rows]
    bits = torch.randint(-2 ** 31, 2 ** 31 - 1, (3000, 8), device="cuda", dtype=torch.int64).to(torch.int32)
    feats = {L: labs.features(L, bits, 8, 3000).clone() for L in (223, 193)}
    torch.cuda.synchronize()
    errors = []
    start = threading.Barrier(len(work) + 2)

    def run(f, n):
        try:
            s = torch.cuda.Stream()
            start.wait()
            with torch.cuda.stream(s):
                for _ in range(n):
                    f(s)
            s.synchronize()
        except Exception as e:  # noqa: BLE001 (reported below)
            errors.append(repr(e))

    def delta(k):
        def f(s):
            out = labs.neighbor_delta(rows[k])
            s.synchronize()
            if not torch.equal(out, want[k]):
                errors.append("rows of work %d differ" % k)
        return f

    def feat(L):
        def f(s):
            out = labs.features(L, bits, 8, 3000)
            s.synchronize()
            if not torch.equal(out, feats[L]):
                errors.append("features of L=%d differ" % L)
        return f

    threads = [threading.Thread(target=run, args=(delta(k), 400)) for k in range(len(work))]
    threads += [threading.Thread(target=run, args=(feat(L), 400)) for L in (223, 193)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors[:3]
