"""Waits of the network kernels that give up (the library's network unit built with no attempts
for one kind of wait, so nothing hangs and nothing faults): the kernels end, every result of the
pass is NaN, and the next pass is as ever."""
from __future__ import annotations

import ctypes
import os
import subprocess

import numpy as np
import pytest
import torch

import paper_2011_00068_gb300 as labs
from oracle import learned as ln
from paper_2011_00068_gb300 import build
from tests.test_gpu_net import net_ws, ptr, random_case

pytestmark = pytest.mark.gpu

# attempts per kind of wait (one takes about 4 us when nothing comes); what a part waits for that
# another part no longer sends is given up after 20000
KINDS = {"weights": {"WEIGHTS": 0, "PRODUCTS": 20000}, "tiles": {"TILES": 0, "PRODUCTS": 20000},
         "products": {"PRODUCTS": 0, "TILES": 20000}}


@pytest.fixture(scope="module")
def variants(tmp_path_factory):
    """One small library per kind of wait, built side by side."""
    out = tmp_path_factory.mktemp("giveup")
    jobs = {}
    for kind, tries in KINDS.items():
        lib = str(out / ("net_%s.so" % kind))
        jobs[kind] = lib, subprocess.Popen(
            [build.nvcc(), "-O3", "-std=c++17", *build.ARCH, "-Xcompiler", "-fPIC", "-shared", "-cudart", "shared", "-I",
             os.path.join(build.ROOT, "include"), *["-DLABS_NET_TRIES_%s=%d" % m for m in tries.items()],
             os.path.join(build.CSRC, "labs_net.cu"), "-o", lib], stdout=subprocess.PIPE, stderr=subprocess.STDOUT)
    libs = {}
    for kind, (lib, job) in jobs.items():
        log = job.communicate()[0].decode()
        assert job.returncode == 0, log
        libs[kind] = ctypes.CDLL(lib)
        for name in ("labs_net_forward", "labs_net_gradients"):
            getattr(libs[kind], name).argtypes = getattr(labs.library(), name).argtypes
    return libs


def passes(lib, n, B, data, ws, wb):
    p, x, t, y, w = data
    sc, rs = torch.zeros((B, n), device="cuda"), torch.zeros(B, device="cuda")
    g, loss = torch.zeros_like(p), torch.zeros(1, device="cuda")
    s = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    assert lib.labs_net_forward(ptr(p), ptr(x), B, n, ptr(sc), ptr(rs), ptr(ws), wb, s) == 0
    assert lib.labs_net_gradients(ptr(p), ptr(x), ptr(t), ptr(y), ptr(w), B, n, ptr(g), ptr(loss), ptr(ws), wb, s) == 0
    torch.cuda.synchronize()
    return sc, rs, g, loss


# several tiles for every tile group, one, and (n = 256) fewer tiles than SMs
@pytest.mark.parametrize("n,B", [(101, 3000), (152, 700), (40, 5), (256, 9)])
@pytest.mark.parametrize("kind", list(KINDS))
def test_a_pass_that_gives_up_returns_nan(variants, kind, n, B):
    params, x = random_case(n, B, seed=n)
    rng = np.random.default_rng(n)
    data = [torch.from_numpy(a).cuda() for a in (ln.flatten(params), x, rng.integers(0, n, B).astype(np.int32),
                                                 rng.standard_normal(B).astype(np.float32), np.ones(B, np.float32))]
    ws, wb = net_ws(n, B)
    want = passes(labs.library(), n, B, data, ws, wb)
    assert all(torch.isfinite(v).all() for v in want)
    sc, rs, g, loss = passes(variants[kind], n, B, data, ws, wb)
    if kind == "tiles":  # (waits of the backward kernels alone)
        assert torch.equal(sc, want[0]) and torch.equal(rs, want[1])
    else:
        assert torch.isnan(sc).all() and torch.isnan(rs).all()
    assert torch.isnan(g).all() and torch.isnan(loss).all()
    again = passes(labs.library(), n, B, data, ws, wb)
    assert torch.equal(again[0], want[0]) and torch.equal(again[1], want[1])
    assert all(torch.isfinite(v).all() for v in again)
