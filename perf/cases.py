"""The workloads that performance work on this library is measured on.

Each case is one call sequence of a user's program through the public entry points
(`Search`, `isl`, `neighbor_delta`, `enumerate_skew`, `features`, `learned.Trainer` and
the C ABI's `labs_net_forward`), at a size taken from the repository's configurations,
benchmark or tests.  `listed()` are the fixed cases, `draw(rng)` gives further ones of
the same families over their whole ranges.  All inputs are synthetic and come from the
seed alone.
"""
from __future__ import annotations

import ctypes
import math

import numpy as np
import torch

import paper_2011_00068_gb300 as labs
from paper_2011_00068_gb300 import _native, learned

NET_SHAPES = [("w1", (64, 16, 7)), ("b1", (64,)), ("w2", (64, 64, 7)), ("b2", (64,)), ("w3", (64, 64, 7)),
              ("b3", (64,)), ("w4", (64, 64)), ("b4", (64,)), ("w5", (64,)), ("b5", (1,)), ("w6", (64,)), ("b6", (1,))]


def listed():
    return [
        # Config 1: the exhaustive optimum of a short length, then few walkers on the same
        # length (whether they reach it), where a step's latency and the launches are all
        # there is; the sequences are read back too.
        {"name": "optimum_41", "kind": "optimum", "L": 41, "walkers": 64, "steps": 1000},
        # Config 2 and the benchmark's workload: the plain walk at full size.
        {"name": "walk_201", "kind": "walk", "L": 201, "walkers": 16384, "steps": 10000},
        # Config 3: all 52 odd lengths of the paper's table in one context (a quarter of
        # its walkers).
        {"name": "walk_mixed_201_303", "kind": "mixed", "L0": 201, "L1": 303, "walkers": 512, "steps": 2000},
        # The scale-up's longer length: one walker per warp.
        {"name": "walk_501", "kind": "walk", "L": 501, "walkers": 16384, "steps": 2000},
        # A long sequence: one walker per CTA (the benchmark's long configuration).
        {"name": "walk_4095", "kind": "walk", "L": 4095, "walkers": 608, "steps": 512},
        # Algorithm 1 as printed: the best-first search on config 2's walkers.
        {"name": "bestfirst_201", "kind": "bestfirst", "L": 201, "walkers": 16384, "steps": 1000},
        # The walk under the PSL objective on the same walkers.
        {"name": "psl_201", "kind": "psl", "L": 201, "walkers": 16384, "steps": 1000},
        # The stateless neighbourhood of a large batch of rows (the benchmark's delta line).
        {"name": "delta_201", "kind": "delta", "L": 201, "rows": 1 << 20},
        # The same for a handful of sequences (a polish step around a few candidates): one
        # small launch.
        {"name": "delta_255_few", "kind": "delta", "L": 255, "rows": 64},
        # ISL of a batch of arbitrary rows (checking or ranking candidate sequences).
        {"name": "isl_255", "kind": "isl", "L": 255, "rows": 1 << 18},
        # Config 4: scoring a batch of states with the proposal network (features, then
        # the forward pass), the batch of one proposal call.
        {"name": "score_255", "kind": "score", "L": 255, "batch": 8192},
        # Config 4: one training step of the proposal network on walk-log records
        # (features, labels, forward, backward, AdamW).
        {"name": "train_255", "kind": "train", "L": 255, "batch": 4096},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _odd(rng, lo, hi):
    return min(hi, max(lo, _log_int(rng, lo, hi) | 1))


def draw(rng):
    kind = rng.choice(["walk", "walk", "walk", "mixed", "long", "bestfirst", "psl", "delta", "delta", "isl", "isl",
                       "optimum", "score", "train"])
    if kind == "walk":
        return {"kind": "walk", "L": _odd(rng, 21, 511), "walkers": _log_int(rng, 16, 16384),
                "steps": _log_int(rng, 256, 4096)}
    if kind == "long":
        L = _odd(rng, 513, 8191)
        return {"kind": "walk", "L": L, "walkers": _log_int(rng, 8, 608), "steps": _log_int(rng, 64, 256)}
    if kind == "mixed":
        L0 = _odd(rng, 101, 255)
        return {"kind": "mixed", "L0": L0, "L1": L0 + 2 * rng.randint(3, 24), "walkers": _log_int(rng, 16, 512),
                "steps": _log_int(rng, 256, 2000)}
    if kind in ("bestfirst", "psl"):
        return {"kind": kind, "L": _odd(rng, 41, 303), "walkers": _log_int(rng, 64, 16384), "steps": _log_int(rng, 128, 1000)}
    if kind == "delta":
        return {"kind": "delta", "L": _odd(rng, 21, 511), "rows": _log_int(rng, 1, 1 << 19)}
    if kind == "isl":
        return {"kind": "isl", "L": _odd(rng, 13, 1023), "rows": _log_int(rng, 1, 1 << 18)}
    if kind == "optimum":
        return {"kind": "optimum", "L": 2 * rng.randint(7, 24) + 1, "walkers": _log_int(rng, 16, 1024),
                "steps": _log_int(rng, 64, 1000)}
    if kind == "score":
        return {"kind": "score", "L": _odd(rng, 41, 511), "batch": _log_int(rng, 1, 8192)}
    return {"kind": "train", "L": _odd(rng, 41, 303), "batch": _log_int(rng, 16, 4096)}


# ---------------------------------------------------------------------- inputs

def _device():
    return torch.device("cuda", torch.cuda.current_device()) if torch.cuda.is_available() else torch.device("cpu")


def _generator(seed, dev):
    g = torch.Generator(device=dev)
    g.manual_seed(int(seed) * 1000003 + 17)
    return g


def _pm1(shape, seed, dev):
    return (1 - 2 * torch.randint(0, 2, shape, device=dev, generator=_generator(seed, dev))).to(torch.int8)


def _expand(x):
    """Skew-symmetric rows [B, 2n-1] of free variables [B, n]: s_{c+j} = (-1)^j s_{c-j}."""
    n = x.shape[1]
    j = torch.arange(1, n, device=x.device)
    sign = torch.where(j % 2 == 1, -1, 1).to(x.dtype)
    return torch.cat([x, x[:, n - 1 - j] * sign], dim=1).contiguous()


def _bits(x):
    """[B, 8] int32 words of free variables [B, n]: bit i set where x_i = -1."""
    B, n = x.shape
    full = torch.zeros((B, 256), dtype=torch.int64, device=x.device)
    full[:, :n] = (x < 0).to(torch.int64)
    w = (full.view(B, 8, 32) << torch.arange(32, device=x.device)).sum(dim=2)
    return torch.where(w >= 2 ** 31, w - 2 ** 32, w).to(torch.int32)


def _autocorrelations(s):
    """C_0 .. C_{L-1} of rows [B, L] (float64, by FFT, rounded to the integers they are)."""
    L = s.shape[1]
    f = torch.fft.rfft(s.to(torch.float64), n=1 << (2 * L - 1).bit_length(), dim=1)
    return torch.fft.irfft(f * f.conj(), dim=1)[:, :L].round()


def _isl(s, chunk=1 << 14):
    return torch.cat([(_autocorrelations(p)[:, 1:] ** 2).sum(dim=1) for p in s.split(chunk)])


def _deltas(s):
    """ISL change of flipping each free variable (and its mirror) of skew-symmetric rows:
    dC_k = -2 s_j (s_{j-k} + s_{j+k}) summed over the flipped positions, pairs of two
    flipped positions left out; float64 [B, n]."""
    B, L = s.shape
    n = (L + 1) // 2
    C = _autocorrelations(s)
    v = torch.zeros((B, 3 * L), dtype=torch.float64, device=s.device)
    v[:, L:2 * L] = s.to(torch.float64)
    out = torch.empty((B, n), dtype=torch.float64, device=s.device)
    for i in range(n):
        dC = torch.zeros((B, L), dtype=torch.float64, device=s.device)
        flipped = {i, L - 1 - i}
        for j in flipped:
            u = v[:, L + j:2 * L + j] + v[:, j + 1:L + j + 1].flip(1)  # s_{j+k} + s_{j-k}, k = 0 .. L-1
            if len(flipped) == 2:
                other = L - 1 - j
                u[:, abs(other - j)] -= v[:, L + other]
            dC -= 2 * v[:, L + j:L + j + 1] * u
        dC[:, 0] = 0
        out[:, i] = (dC * (2 * C + dC)).sum(dim=1)
    return out


def _net_params(seed, dev):
    """Network parameters of the size a trained network has, in the library's order."""
    rng = np.random.default_rng(seed + 7919)
    parts = []
    for name, shape in NET_SHAPES:
        fan = int(np.prod(shape[1:])) if len(shape) > 1 else 64
        scale = 0.05 if name.startswith("b") else math.sqrt(2.0 / fan)
        parts.append((rng.standard_normal(shape) * scale).astype(np.float32).ravel())
    return torch.from_numpy(np.concatenate(parts)).to(dev)


def _records(L, batch, seed, dev):
    """Walk-log records (uint8 [batch, 64]) of random states: the state's bits and ISL, a
    first flip, and the lowest ISL of the steps that followed (below the start's in most)."""
    n = (L + 1) // 2
    x = _pm1((batch, n), seed, dev)
    isl = _isl(_expand(x)).to(torch.int64)
    g = _generator(seed + 1, dev)
    first = torch.randint(0, n, (batch,), device=dev, generator=g)
    low = torch.rand(batch, device=dev, generator=g) * 0.75 + 0.3
    low = torch.minimum(isl, (isl.to(torch.float64) * low).to(torch.int64).clamp(min=1))
    rec = torch.zeros((batch, 16), dtype=torch.int32, device=dev)
    rec[:, :8] = _bits(x)
    rec[:, 8] = isl.to(torch.int32)
    rec[:, 9] = first.to(torch.int32)
    rec[:, 10] = low.to(torch.int32)
    rec[:, 11] = L
    rec[:, 12] = torch.arange(batch, device=dev, dtype=torch.int32)
    return x, rec


def _counts(case):
    Ls = list(range(case["L0"], case["L1"] + 1, 2))
    return Ls, [case["walkers"]] * len(Ls)


def _ptr(t):
    return ctypes.c_void_p(t.data_ptr())


def prepare(case, seed):
    kind, dev = case["kind"], _device()
    if kind in ("walk", "optimum", "bestfirst", "psl", "mixed"):
        if kind == "mixed":
            Ls, counts = _counts(case)
            s = labs.Search(Ls, counts, int(seed))
        elif kind == "psl":
            s = labs.Search(case["L"], case["walkers"], int(seed), objective="psl")
        else:
            flags = _native.LABS_FLAG_BEST_FIRST if kind == "bestfirst" else 0
            s = labs.Search(case["L"], case["walkers"], int(seed), flags=flags)
        return {"case": case, "search": s}
    if kind == "delta":
        return {"case": case, "rows": _expand(_pm1((case["rows"], (case["L"] + 1) // 2), seed, dev))}
    if kind == "isl":
        return {"case": case, "rows": _pm1((case["rows"], case["L"]), seed, dev)}
    L, B = case["L"], case["batch"]
    n = (L + 1) // 2
    x, rec = _records(L, B, seed, dev)
    params = _net_params(seed, dev)
    if kind == "score":
        nbytes = ctypes.c_size_t()
        rc = labs.library().labs_net_sizes(n, B, None, ctypes.byref(nbytes))
        if rc:
            raise RuntimeError("labs_net_sizes: %d" % rc)
        return {"case": case, "bits": rec[:, :8].contiguous(), "params": params,
                "scores": torch.empty((B, n), device=dev), "restart": torch.empty(B, device=dev),
                "ws": torch.empty(int(nbytes.value), dtype=torch.uint8, device=dev)}
    # a run some thousand steps in: moments filled, bias corrections near their ends
    t = learned.Trainer(L, B, int(seed))
    g = _generator(seed + 2, dev)
    t.params.copy_(params)
    t.m.copy_(torch.randn(params.shape, device=dev, generator=g) * 1e-3)
    t.v.copy_((torch.rand(params.shape, device=dev, generator=g) + 0.5) * 1e-5)
    t.t = 4000
    return {"case": case, "trainer": t, "records": rec.view(torch.uint8).view(B, 64)}


# ------------------------------------------------------------------------ passes

def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind in ("walk", "optimum", "bestfirst", "psl", "mixed"):
        # the whole search: fresh starts, the steps, every walker's results, the best one
        s = state["search"]
        s.reset()
        s.walk(case["steps"])
        r = s.results(seqs=kind == "optimum")
        b = s.best()
        if kind == "optimum":
            least, count, first = labs.enumerate_skew(case["L"])
            r["optimum"] = {"isl": least, "count": count, "first": first}
        r["best"] = {k: b[k] for k in ("L", "isl", "seq")}
        if kind == "psl":
            r["best"]["psl"] = b["psl"]
        return r
    if kind == "delta":
        return labs.neighbor_delta(state["rows"])
    if kind == "isl":
        return labs.isl(state["rows"])
    L, B = case["L"], case["batch"]
    if kind == "score":
        x = labs.features(L, state["bits"], 8, B)
        s = torch.cuda.current_stream()
        rc = labs.library().labs_net_forward(_ptr(state["params"]), _ptr(x), B, (L + 1) // 2, _ptr(state["scores"]),
                                             _ptr(state["restart"]), _ptr(state["ws"]), state["ws"].numel(),
                                             ctypes.c_void_p(s.cuda_stream))
        if rc:
            raise RuntimeError("labs_net_forward: %d" % rc)
        return {"features": x, "scores": state["scores"], "restart": state["restart"]}
    t = state["trainer"]
    loss = t.step(state["records"])
    return {"loss": loss, "grads": t.grads, "params": t.params, "m": t.m, "v": t.v}


# ------------------------------------------------------- what a pass cannot do without

def work(case):
    """Bytes: inputs read once, outputs written once (a walker step: one probe and one
    insertion of 8 bytes in its visited set).  Flops: two per lag term of a neighbourhood
    (n - 1 terms per flip) or per term of an autocorrelation, and the network's products."""
    kind = case["kind"]
    if kind == "mixed":
        Ls, counts = _counts(case)
        flops = sum(2 * c * case["steps"] * ((L + 1) // 2) * ((L - 1) // 2) for L, c in zip(Ls, counts))
        return {"bytes": sum(counts) * (16 * case["steps"] + 16), "flops": flops}
    L = case["L"]
    n = (L + 1) // 2
    if kind in ("walk", "optimum", "bestfirst", "psl"):
        w = case["walkers"] * case["steps"]
        flops = (2 if kind != "psl" else 5) * n * (n - 1) * w
        if kind == "optimum":
            flops += 4 * (n - 1) * 2 ** (n - 1)  # every assignment's even lags, from its neighbour's
        return {"bytes": 16 * w + 16 * case["walkers"], "flops": flops}
    if kind == "delta":
        return {"bytes": case["rows"] * (L + 4 * n), "flops": 2 * n * (n - 1) * case["rows"]}
    if kind == "isl":
        return {"bytes": case["rows"] * (L + 4), "flops": L * (L - 1) * case["rows"]}
    B, macs = case["batch"], n * (3 * 7 * 64 + 2 * 64 * 7 * 64 + 64 * 64 + 2 * 64)
    if kind == "score":
        return {"bytes": B * (32 + 16 * n + 4) + 4 * 68994, "flops": 2 * B * macs}
    return {"bytes": B * 64 + 4 * 68994 * 7, "flops": 6 * B * macs}


# ------------------------------------------------------------------- 64-bit results

def _net_forward(p, x):
    """Scores [B, n], restart scores [B] and the activations, in p's type."""
    F = torch.nn.functional
    a = [torch.cat([x, x.new_zeros((x.shape[0], 13, x.shape[2]))], dim=1)]
    for l in ("1", "2", "3"):
        # one product per tap (the library's own double convolutions are far slower)
        pad = F.pad(a[-1], (3, 3))
        n = x.shape[2]
        y = sum(torch.einsum("oc,bcp->bop", p["w" + l][:, :, k], pad[:, :, k:k + n]) for k in range(7))
        a.append(torch.relu(y + p["b" + l][None, :, None]))
    h = torch.relu(torch.einsum("jc,bcp->bjp", p["w4"], a[3]) + p["b4"][None, :, None])
    score = torch.einsum("j,bjp->bp", p["w5"], h) + p["b5"]
    restart = a[3].mean(dim=2) @ p["w6"] + p["b6"]
    return score, restart


def _unflatten(flat):
    p, off = {}, 0
    for name, shape in NET_SHAPES:
        k = int(np.prod(shape))
        p[name] = flat[off:off + k].view(shape)
        off += k
    return p


def _features(x, L):
    n = x.shape[1]
    s = _expand(x)
    C = _autocorrelations(s)
    d = torch.cat([_deltas(q) for q in s.split(1 << 14)])
    f = torch.zeros((x.shape[0], 3, n), dtype=torch.float64, device=x.device)
    f[:, 0] = x.to(torch.float64)
    k = torch.arange(1, n, device=x.device)
    f[:, 1, :n - 1] = C[:, 2 * k] / math.sqrt(L)
    f[:, 2] = d / (8 * L)
    return f


def exact(case, seed):
    kind, dev = case["kind"], _device()
    if kind == "isl":
        return _isl(_pm1((case["rows"], case["L"]), seed, dev))
    if kind == "delta":
        s = _expand(_pm1((case["rows"], (case["L"] + 1) // 2), seed, dev))
        return torch.cat([_deltas(q) for q in s.split(1 << 17)])
    if kind not in ("score", "train"):
        return None  # a search: its outputs are whole numbers with no closed form
    L, B = case["L"], case["batch"]
    n = (L + 1) // 2
    x, rec = _records(L, B, seed, dev)
    feats = _features(x, L)
    flat = _net_params(seed, dev).to(torch.float64)
    if kind == "score":
        with torch.no_grad():
            out = [_net_forward(_unflatten(flat), q) for q in feats.split(1024)]
        return {"features": feats, "scores": torch.cat([o[0] for o in out]), "restart": torch.cat([o[1] for o in out])}
    target, isl, low = rec[:, 9].long(), rec[:, 8], rec[:, 10]
    wf = (low < isl).to(torch.float64)
    y = L * L / (2.0 * low.to(torch.float64)) / 8.0
    flat.requires_grad_(True)
    total = 0.0
    for q in torch.arange(B, device=dev).split(512):
        score, restart = _net_forward(_unflatten(flat), feats[q])
        ce = torch.nn.functional.cross_entropy(score, target[q], reduction="none")
        loss = (wf[q] * ce + 0.5 * (restart - y[q]) ** 2).sum() / B
        loss.backward()
        total += float(loss.detach())
    grad = flat.grad
    prm = flat.detach()
    g = _generator(seed + 2, dev)
    m = torch.randn(prm.shape, device=dev, generator=g).to(torch.float32) * 1e-3
    v = (torch.rand(prm.shape, device=dev, generator=g) + 0.5) * 1e-5
    m = 0.9 * m.to(torch.float64) + 0.1 * grad
    v = 0.999 * v.to(torch.float64) + 0.001 * grad * grad
    decay = torch.cat([torch.full((int(np.prod(s)),), 0.0 if nm.startswith("b") else 0.01, dtype=torch.float64, device=dev)
                       for nm, s in NET_SHAPES])
    mh, vh = m / (1 - 0.9 ** 4001), v / (1 - 0.999 ** 4001)
    new = prm - 1e-3 * (mh / (vh.sqrt() + 1e-8) + decay * prm)
    return {"loss": torch.tensor([total], dtype=torch.float64), "grads": grad, "params": new, "m": m, "v": v}
