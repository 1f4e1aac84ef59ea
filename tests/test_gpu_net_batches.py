"""Batches in which a CTA of the network kernels takes several tiles: 256-row tiles (n > 128), the
second and third turn of the backward kernels' barriers (n <= 128), and more states than one
pass of the network's input kernel holds."""
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


@pytest.mark.parametrize("n,B", [(152, 1200), (256, 1000)])
def test_forward_several_tiles(n, B):
    params, x = random_case(n, B, seed=n)
    sc, rs = gpu_forward(ln.flatten(params), x)
    net, xo = ln.Net(True), oracle_x(x)
    rng = np.random.default_rng(n)
    for b in sorted(set(rng.choice(B, 12, replace=False).tolist()) | {0, B - 1}):
        fw = net.forward(params, xo[b])
        assert_close(sc[b], fw["score"], "score of sample %d" % b)
        terms = float(np.abs(fw["W"]["w6"] * fw["pooled"]).sum() + abs(params["b6"][0]))
        assert_close(rs[b], fw["restart"], "restart score of sample %d" % b, scale=terms)


@pytest.mark.parametrize("n,B", [(152, 1200), (256, 700), (101, 3100)])
def test_gradients_several_tiles(n, B):
    params, x = random_case(n, B, seed=200 + n)
    rng = np.random.default_rng(n)
    target = rng.integers(0, n, B).astype(np.int32)
    y = rng.standard_normal(B).astype(np.float32)
    wf = (rng.random(B) < 0.7).astype(np.float32)
    ws, wb = net_ws(n, B)
    p = torch.from_numpy(ln.flatten(params)).cuda()
    g, loss = torch.empty_like(p), torch.zeros(1, device="cuda")
    s = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    xd, td, yd, wd = (torch.from_numpy(a).cuda() for a in (x, target, y, wf))
    assert labs.library().labs_net_gradients(ptr(p), ptr(xd), ptr(td), ptr(yd), ptr(wd), B, n, ptr(g), ptr(loss),
                                             ptr(ws), wb, s) == 0
    torch.cuda.synchronize()
    gpu = ln.unflatten(g.cpu().numpy())
    oloss, og = ln.Net(True).batch_loss_and_grads(params, list(oracle_x(x)), target, y, wf)
    assert_close(loss.item(), oloss, "loss", scale=0.0)
    for name, _ in ln.PARAM_SHAPES:
        assert_close(gpu[name], og[name], "gradient of " + name, scale=1e-3 if name == "b5" else None)


@pytest.mark.parametrize("L,stride", [(41, 8), (255, 16), (401, 8)])
def test_features_of_many_states(L, stride):
    B, n = 40001, (L + 1) // 2
    g = torch.Generator(device="cuda")
    g.manual_seed(L)
    bits = torch.randint(-2 ** 31, 2 ** 31 - 1, (B, stride), device="cuda", dtype=torch.int64, generator=g).to(torch.int32)
    got = labs.features(L, bits, stride, B)
    for first in range(0, B, 1000):  # the same states, a few at a time
        part = bits[first:first + 1000].contiguous()
        assert torch.equal(got[first:first + 1000], labs.features(L, part, stride, part.shape[0]))
