"""The network's tile kernels at the edges of a tile: several samples per tile (short n),
a last tile that is partly empty, one sample filling 128 rows, and the 256-row tiles
above n = 128, forward and gradients against oracle/learned.py element by element (the
bound of tests/nettol.py)."""
from __future__ import annotations

import ctypes

import numpy as np
import pytest
import torch

import paper_2011_00068_gb300 as labs
from oracle import learned as ln
from tests.nettol import assert_close
from tests.test_gpu_net import gpu_forward, net_ws, oracle_x, ptr, random_case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,B", [(2, 1), (2, 27), (5, 70), (40, 7), (63, 9), (125, 3), (127, 2), (128, 1), (129, 2),
                                 (152, 3), (256, 2)])
def test_tiles_match_oracle(n, B):
    params, x = random_case(n, B, seed=1000 + n)
    flat = ln.flatten(params)
    sc, rs = gpu_forward(flat, x)
    net, xo = ln.Net(True), oracle_x(x)
    for b in range(B):
        fw = net.forward(params, xo[b])
        assert_close(sc[b], fw["score"], "score of sample %d" % b)
        terms = float(np.abs(fw["W"]["w6"] * fw["pooled"]).sum() + abs(params["b6"][0]))
        assert_close(rs[b], fw["restart"], "restart score of sample %d" % b, scale=terms)

    rng = np.random.default_rng(n)
    target = rng.integers(0, n, B).astype(np.int32)
    y = rng.standard_normal(B).astype(np.float32)
    wf = (rng.random(B) < 0.7).astype(np.float32)
    wf[0] = 1.0
    ws, wb = net_ws(n, B)
    ws.fill_(0xFF)  # nothing may depend on what the workspace held (0xFF bytes are NaNs)
    p = torch.from_numpy(flat).cuda()
    g = torch.full_like(p, float("nan"))
    loss = torch.zeros(1, device="cuda")
    xd, td, yd, wd = (torch.from_numpy(a).cuda() for a in (x, target, y, wf))
    s = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    assert labs.library().labs_net_gradients(ptr(p), ptr(xd), ptr(td), ptr(yd), ptr(wd), B, n, ptr(g), ptr(loss),
                                             ptr(ws), wb, s) == 0
    torch.cuda.synchronize()
    gpu = ln.unflatten(g.cpu().numpy())
    oloss, og = net.batch_loss_and_grads(params, list(xo), target, y, wf)
    assert_close(loss.item(), oloss, "loss", scale=0.0)
    for name, _ in ln.PARAM_SHAPES:
        assert_close(gpu[name], og[name], "gradient of " + name, scale=1e-3 if name == "b5" else None)
