"""The proposal network's inputs (labs_features) at the edges of the row kernels: lane blocks,
words per class, odd counts, strides, and set bits above n that are not part of the state."""
from __future__ import annotations

import numpy as np
import pytest
import torch

import labs_inputs
import oracle
import paper_2011_00068_gb300 as labs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L", [3, 5, 31, 33, 63, 65, 95, 127, 129, 161, 193, 225, 255, 257, 319, 321, 385, 449, 509, 511])
@pytest.mark.parametrize("stride", [8, 11])
def test_features_of_every_kernel(L, stride):
    n, B = (L + 1) // 2, 5
    xs = labs_inputs.random_free_vars(B, L, seed=L)
    bits = np.full((B, stride), 0xDEADBEEF, np.uint32)
    for b, x in enumerate(xs):
        v = sum(1 << i for i in range(n) if x[i] < 0) | (~0 << n & (1 << 256) - 1 if b == 1 else 0)
        for k in range(8):
            bits[b, k] = v >> (32 * k) & 0xFFFFFFFF
    got = labs.features(L, torch.from_numpy(bits.view(np.int32)).cuda(), stride, B).cpu().numpy()
    for b, x in enumerate(xs):
        row = oracle.skew_expand(x, L).astype(np.int64)
        C = np.array([(row[:L - 2 * m] * row[2 * m:]).sum() for m in range(1, n)] + [0])
        C[-1] = 0
        want = np.stack([row[:n].astype(np.float32), C.astype(np.float32) / np.sqrt(np.float32(L)),
                         oracle.neighbor_delta(oracle.skew_expand(x, L)).astype(np.float32) / np.float32(8 * L)])
        assert np.array_equal(got[b].reshape(3, n), want), b
