"""The chains of products that W4's gradient is added up in: two accumulators per SM at every
length, taken in turn by the tiles of an SM.  A tensor-core accumulator rounds every addition
toward zero, so what small products lose beside large ones shows which tiles share one.

Everything but those additions is exact here.  One position per sample is marked (feature 0),
the convolutions pass the mark on, unit 0 of the MLP is 1 elsewhere and unit 1 is 1 at the mark,
so the scores are all equal, the softmax is 1/n (n a power of two) and dh is w_b / (n B) at the
n - 1 unmarked positions, a power of two.  Then dW4[0][c] = b3_c sum_b w_b (n - 1) / (n B), with
8-bit b3_c.  The samples of SM 0 alone have weights: its first tile 2^20, every second one after
it 1.  Beside the first tile's sum a later one's products (below half a unit in the last place,
16 rows at a time) vanish; by themselves they are exact, and the only rounding left is that of
the last addition of two partial sums: 2^-24 of the result (the bound is twice that)."""
from __future__ import annotations

import ctypes

import numpy as np
import pytest
import torch

import paper_2011_00068_gb300 as labs
from oracle import learned as ln
from tests.test_gpu_net import net_ws, ptr

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [128, 256])
def test_w4_gradient_keeps_small_tiles(n):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    B = 2048  # one sample per tile: about 13 tiles of SM 0
    p = {name: np.zeros(shape, np.float32) for name, shape in ln.PARAM_SHAPES}
    for w in ("W1", "W2", "W3"):
        p[w][0, 0, 3] = 1.0
    b3 = (128 + (37 * np.arange(64)) % 128 | 1).astype(np.float32) / 128
    p["b3"][1:] = b3[1:]
    p["W4"][0, 0], p["b4"][0] = -1.0, 1.0
    p["W4"][1, 0] = 1.0
    p["w5"].reshape(-1)[:2] = 1.0
    rng = np.random.default_rng(3)
    target = rng.integers(0, n, B).astype(np.int32)
    x = np.zeros((B, 3, n), np.float32)
    x[np.arange(B), 0, target] = 1.0
    wf = np.zeros(B, np.float32)
    wf[0] = 2.0 ** 20
    wf[sms::2 * sms] = 1.0
    assert np.count_nonzero(wf) > 5
    ws, wb = net_ws(n, B)
    prm = torch.from_numpy(ln.flatten(p)).cuda()
    g, loss = torch.empty_like(prm), torch.zeros(1, device="cuda")
    xd, td, wd = (torch.from_numpy(a).cuda() for a in (x, target, wf))
    yd = torch.zeros(B, device="cuda")
    s = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    assert labs.library().labs_net_gradients(ptr(prm), ptr(xd), ptr(td), ptr(yd), ptr(wd), B, n, ptr(g), ptr(loss),
                                             ptr(ws), wb, s) == 0
    torch.cuda.synchronize()
    got = ln.unflatten(g.cpu().numpy())["W4"][0].astype(np.float64)
    want = b3.astype(np.float64) * wf.astype(np.float64).sum() * (n - 1) / (n * B)
    assert got[0] == 0.0
    err = np.abs(got[1:] - want[1:]) / want[1:]
    print("n=%d: largest relative error %.3g" % (n, err.max()))
    assert err.max() <= 2.0 ** -23
