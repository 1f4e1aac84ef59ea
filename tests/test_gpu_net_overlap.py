"""Network results that overlap the pass's inputs (scores written over the states, gradients over
the labels or the parameters): the same as apart from them."""
from __future__ import annotations

import ctypes

import numpy as np
import pytest
import torch

import paper_2011_00068_gb300 as labs
from oracle import learned as ln
from tests.test_gpu_net import net_ws, ptr, random_case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,B", [(41, 3000), (128, 2000), (152, 1000)])
@pytest.mark.parametrize("place", ["begin", "end"])
def test_results_over_inputs(n, B, place):
    params, x = random_case(n, B, seed=n)
    rng = np.random.default_rng(n)
    flat = ln.flatten(params)
    N = flat.size
    s = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    lib = labs.library()
    ws, wb = net_ws(n, B)
    p, xd = torch.from_numpy(flat).cuda(), torch.from_numpy(x).cuda()
    sc, rs = torch.empty((B, n), device="cuda"), torch.empty(B, device="cuda")
    assert lib.labs_net_forward(ptr(p), ptr(xd), B, n, ptr(sc), ptr(rs), ptr(ws), wb, s) == 0

    over = xd.clone().view(-1)
    at = 0 if place == "begin" else over.numel() - B * n - B
    o_sc, o_rs = over[at:at + B * n], over[at + B * n:at + B * n + B]
    assert lib.labs_net_forward(ptr(p), ptr(over), B, n, ptr(o_sc), ptr(o_rs), ptr(ws), wb, s) == 0
    torch.cuda.synchronize()
    assert torch.equal(o_sc.view(B, n), sc) and torch.equal(o_rs, rs)

    t, y, w = (torch.from_numpy(a).cuda() for a in (rng.integers(0, n, B).astype(np.int32),
                                                    rng.standard_normal(B).astype(np.float32), np.ones(B, np.float32)))
    g, loss = torch.empty_like(p), torch.zeros(1, device="cuda")
    assert lib.labs_net_gradients(ptr(p), ptr(xd), ptr(t), ptr(y), ptr(w), B, n, ptr(g), ptr(loss), ptr(ws), wb, s) == 0
    torch.cuda.synchronize()
    scale = float(g.abs().max())

    def check(got, what):
        # the bias gradients' float32 additions come in any order (about 1e-6 of the largest)
        torch.cuda.synchronize()
        assert torch.isfinite(got).all(), what
        assert float((got - g).abs().max()) <= 1e-4 * scale, what

    over = xd.clone().view(-1)
    o_g = over[:N] if place == "begin" else over[-N:]
    assert lib.labs_net_gradients(ptr(p), ptr(over), ptr(t), ptr(y), ptr(w), B, n, ptr(o_g), None, ptr(ws), wb, s) == 0
    check(o_g, "over the states")
    o_p = p.clone()
    assert lib.labs_net_gradients(ptr(o_p), ptr(xd), ptr(t), ptr(y), ptr(w), B, n, ptr(o_p), None, ptr(ws), wb, s) == 0
    check(o_p, "over the parameters")
    o_y = torch.zeros(N + B, device="cuda")
    o_y[:B] = y
    assert lib.labs_net_gradients(ptr(p), ptr(xd), ptr(t), ptr(o_y), ptr(w), B, n, ptr(o_y), None, ptr(ws), wb, s) == 0
    check(o_y[:N], "over the labels")
