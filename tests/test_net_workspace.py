"""The network's workspace off a 16-byte boundary (a slice of a larger buffer) is refused on
the host: the kernels' bulk copies and 16-byte stores need the boundary.  No kernel is
launched, so the addresses are only numbers and no GPU is needed for the network's calls."""
from __future__ import annotations

import ctypes

import pytest
import torch

import paper_2011_00068_gb300 as labs
from paper_2011_00068_gb300 import _native, build


@pytest.fixture(scope="module")
def lib():
    try:
        build.nvcc()
    except RuntimeError:
        pytest.skip("no nvcc in this environment")
    return _native.load()


@pytest.mark.parametrize("off", [1, 2, 4, 8, 12])
@pytest.mark.parametrize("n,B", [(40, 7), (152, 3)])
def test_unaligned_workspace_is_refused(lib, n, B, off):
    nbytes = ctypes.c_size_t()
    assert lib.labs_net_sizes(n, B, None, ctypes.byref(nbytes)) == 0
    at = lambda k: ctypes.c_void_p((k << 32) + 0x1000)  # never read: the call is refused first
    ws = ctypes.c_void_p((9 << 32) + off)
    assert lib.labs_net_forward(at(1), at(2), B, n, at(3), at(4), ws, nbytes.value, None) == _native.LABS_EINVAL
    assert lib.labs_net_gradients(at(1), at(2), at(3), at(4), at(5), B, n, at(6), at(7), ws, nbytes.value,
                                  None) == _native.LABS_EINVAL
    # a short workspace is still the first complaint
    assert lib.labs_net_forward(at(1), at(2), B, n, at(3), at(4), ws, nbytes.value - 1, None) == _native.LABS_ENOMEM


@pytest.mark.gpu
@pytest.mark.parametrize("flags", [_native.LABS_FLAG_LEARNED, _native.LABS_FLAG_LEARNED_RESTARTS])
def test_unaligned_learned_workspace_is_refused(flags):
    s = labs.Search(41, 8, 1, tabu_log2=8, flags=flags)
    nbytes = ctypes.c_size_t()
    assert s.lib.labs_learned_workspace_bytes(s.ctx, 4, ctypes.byref(nbytes)) == 0
    buf = torch.empty(nbytes.value + 16, dtype=torch.uint8, device="cuda")
    params = torch.zeros(_param_count(), device="cuda")
    for off in (4, 8):
        rc = s.lib.labs_learned(s.ctx, ctypes.c_void_p(params.data_ptr()), 0, 4,
                                ctypes.c_void_p(buf.data_ptr() + off), nbytes.value)
        assert rc == _native.LABS_EINVAL
    assert b"aligned" in s.lib.labs_last_error(s.ctx)
    s.walk(16)  # the walk goes on without the network
    s.sync()
    s.close()


@pytest.mark.gpu
@pytest.mark.parametrize("n", [2, 41, 101, 128, 152, 256])
def test_small_batches_need_small_workspaces(n):
    """A batch's workspace holds what its own tiles use (a few MB for one state, where the
    partial sums of every CTA that the GPU could run take 80 MB), and never shrinks with the
    batch, so that one sized for the largest batch serves all."""
    sizes = []
    for B in (1, 2, 8, 64, 151, 152, 153, 303, 304, 305, 1000, 4096, 8192):
        nbytes = ctypes.c_size_t()
        assert labs.library().labs_net_sizes(n, B, None, ctypes.byref(nbytes)) == 0
        sizes.append(nbytes.value)
    assert sizes[0] < 2 << 20 and sizes[2] < 12 << 20
    assert sizes == sorted(sizes)


def _param_count():
    k = ctypes.c_size_t()
    assert labs.library().labs_net_sizes(21, 1, ctypes.byref(k), None) == 0
    return int(k.value)
