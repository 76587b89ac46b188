"""The work whose speed counts: transforms as programs ask for them through `Plan`.

A case is one plan and one `Plan.execute` on a cube that lies in device memory.  The plan, the input and the output
buffer are what such a program keeps between transforms, so `prepare` makes them and `run` is the call alone.
"""
import math

import numpy as np
import torch

import paper_2002_03260_b200 as dft
from paper_2002_03260_b200 import inputs

_MODES = {"kdft": dft.DFT3D_KDFT, "fft": dft.DFT3D_FFT, "auto": dft.DFT3D_AUTO}
_FFT_LENGTHS = (256, 512, 1024, 2048)


def _case(name, shape, mode, sign=-1, nodes="", split="", axes="012", dist="normal"):
    """nodes: which axes have nonuniform nodes ("012", "1", ...), with a leading "o" for nodes on the output index, "s"
    for the inverse as a solve; split: "" (the default), "tf32"; axes: the transformed axes; dist: the values."""
    c = {"n0": shape[0], "n1": shape[1], "n2": shape[2], "mode": mode, "sign": sign, "nodes": nodes, "split": split,
         "axes": axes, "dist": dist}
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest cube in use: launches and latency are all of it
        _case("kdft-64", (64, 64, 64), "kdft", dist="uniform"),
        # lengths that fit no tile (not even multiples of four): the TF32 pieces
        _case("kdft-ragged", (100, 66, 250), "kdft"),
        # the ordinary dense transform, in the direction back from the spectrum (scaled by 1/n per axis)
        _case("kdft-512-inverse", (512, 512, 512), "kdft", sign=+1),
        # the largest dense cube that is transformed in one call and still leaves room for the program's own data
        _case("kdft-1024", (1024, 1024, 1024), "kdft", dist="uniform"),
        # samples at sorted random positions on all three axes
        _case("nonuniform-256", (256, 256, 256), "kdft", nodes="012"),
        # jittered samples back from their spectrum: the per-axis systems solved, one axis uniform
        _case("nonuniform-solve", (64, 128, 192), "kdft", sign=+1, nodes="s02"),
        # a cube that almost fits L2, two-factor lengths
        _case("fft-256-inverse", (256, 256, 256), "fft", sign=+1),
        # the headline cube in the FFT formulation
        _case("fft-1024", (1024, 1024, 1024), "fft", dist="uniform"),
        # the long axes of the largest cube (2048 points), slabs of it
        _case("fft-2048-slab", (256, 2048, 2048), "fft"),
        # TF32 pieces on request (full relative precision on every element)
        _case("fft-512-tf32", (512, 256, 512), "fft", split="tf32"),
        # one 8192 x 8192 image: a two-dimensional transform
        _case("fft-2d-8192", (1, 8192, 8192), "fft", axes="12"),
        # one axis has no FFT length: the formulation is chosen per axis
        _case("auto-mixed", (200, 512, 1024), "auto"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _cost(c):
    """Real multiply-adds of the dense products (KDFT axes), plus the points moved: what bounds a drawn case."""
    n = (c["n0"], c["n1"], c["n2"])
    p = n[0] * n[1] * n[2]
    dense = sum(n[int(a)] for a in c["axes"]) if c["mode"] != "fft" else 0
    return p * (dense + 512)


def draw(rng):
    largest = _cost(_case("", (1024, 1024, 1024), "kdft"))
    while True:
        kind = rng.choice(("kdft", "kdft", "nodes", "fft", "fft", "planes", "lines", "auto"))
        sign = rng.choice((-1, +1))
        dist = rng.choice(("normal", "uniform"))
        split = "tf32" if rng.random() < 0.15 else ""
        if kind in ("kdft", "nodes"):
            top = 1024 if kind == "kdft" else 512
            n = [_log_int(rng, 24, top) for _ in range(3)]
            if rng.random() < 0.7:
                n = [max(4, (v + 2) // 4 * 4) for v in n]      # the lengths that keep the default pieces
            n[2] += n[2] % 2                                   # the last axis is always even
            nodes = ""
            if kind == "nodes":
                nodes = ("o" if rng.random() < 0.3 else "") + rng.choice(("012", "012", "0", "1", "2", "01", "12"))
            c = _case("", n, "kdft", sign, nodes, split, "012", dist)
        elif kind == "fft":
            c = _case("", [rng.choice(_FFT_LENGTHS) for _ in range(3)], "fft", sign, "", split, "012", dist)
        elif kind == "planes":     # a batch of two-dimensional transforms, in either formulation
            mode = rng.choice(("kdft", "fft"))
            if mode == "fft":
                n = [_log_int(rng, 3, 300), rng.choice(_FFT_LENGTHS), rng.choice(_FFT_LENGTHS)]
            else:
                n = [_log_int(rng, 3, 300), _log_int(rng, 8, 192) * 4, _log_int(rng, 8, 192) * 4]
            c = _case("", n, mode, sign, "", split, "12", dist)
        elif kind == "lines":      # a batch of one-dimensional transforms along the last or the middle axis
            n = [_log_int(rng, 3, 500), 64 * _log_int(rng, 1, 16), rng.choice(_FFT_LENGTHS)]
            c = _case("", n, "fft", sign, "", split, "2", dist)
            if rng.random() < 0.5:
                c["n1"], c["n2"], c["axes"] = c["n2"], c["n1"], "1"
        else:
            n = [_log_int(rng, 24, 400), rng.choice(_FFT_LENGTHS), rng.choice(_FFT_LENGTHS)]
            n[0] = max(4, n[0] // 4 * 4)
            c = _case("", n, "auto", sign, rng.choice(("", "", "1", "2")), split, "012", dist)
        points = c["n0"] * c["n1"] * c["n2"]
        if points <= 1 << 30 and _cost(c) <= largest:
            return c


def _nodes(case, seed):
    spec = case["nodes"]
    if not spec:
        return None
    shape = (case["n0"], case["n1"], case["n2"])
    which = [int(a) for a in spec.lstrip("os")]
    if spec[0] == "s":             # a solvable system: the uniform grid, every sample moved by less than a third of a step
        r = np.random.default_rng(seed + 1)
        full = [(np.arange(n) + 0.3 * r.uniform(-1.0, 1.0, n)) / n for n in shape]
    else:
        full = inputs.sorted_nodes(shape, seed + 1)
    return [full[a] if a in which else None for a in range(3)]


def prepare(case, seed):
    shape = (case["n0"], case["n1"], case["n2"])
    flags = dft.DFT3D_SPLIT_TF32 if case["split"] == "tf32" else 0
    if case["nodes"].startswith("o"):
        flags |= dft.DFT3D_NODES_ON_OUTPUT
    if case["nodes"].startswith("s"):
        flags |= dft.DFT3D_INVERSE_SOLVE
    plan = dft.Plan(*shape, mode=_MODES[case["mode"]], sign=case["sign"], nodes=_nodes(case, seed), flags=flags,
                    axes=[int(a) for a in case["axes"]])
    x = inputs.cube(shape, case["dist"], seed, device="cuda")
    return plan, x, torch.empty_like(x)


def run(state):
    plan, x, out = state
    return plan(x, out)


def work(case):
    """Input read once, output written once.  Operations: 5 n log2(n) per line of a uniform axis; a nonuniform axis is
    a product with an n x n matrix, of which its conjugate symmetry leaves two real n x n/2 products per real line."""
    n = (case["n0"], case["n1"], case["n2"])
    p = float(n[0] * n[1] * n[2])
    uneven = case["nodes"].lstrip("os")
    flops = sum(p * (4.0 * n[int(a)] if a in uneven else 5.0 * math.log2(max(2, n[int(a)]))) for a in case["axes"])
    return {"bytes": 16.0 * p, "flops": flops}


def tolerance(case):
    """Dense products in 32-bit sums: up to 2.7e-6 over three axes against 64-bit results.  FFT: 2e-7 per axis (fp16
    pieces), 6e-7 (TF32 pieces)."""
    if case["mode"] == "fft":
        return {"rel": 4e-6 if case["split"] == "tf32" else 2e-6}
    return {"rel": 1e-5}


def exact(case, seed):
    """The same transform in 64 bits: numpy's definition of the matrices, torch's complex128 products and transforms."""
    shape = (case["n0"], case["n1"], case["n2"])
    x = inputs.cube(shape, case["dist"], seed, device="cuda").to(torch.complex128)
    nodes = _nodes(case, seed) or [None, None, None]
    sign, spec = case["sign"], case["nodes"]
    for a in (int(c) for c in case["axes"]):
        if nodes[a] is None:
            x = torch.fft.fft(x, dim=a) if sign < 0 else torch.fft.ifft(x, dim=a)
            continue
        k, t = np.arange(shape[a]), np.asarray(nodes[a])
        phase = np.outer(t, k) if spec[0] == "o" else np.outer(k, t)
        if spec[0] == "s":
            m = np.linalg.inv(np.exp(-2j * np.pi * phase))
        else:
            m = np.exp(sign * 2j * np.pi * phase) / (shape[a] if sign > 0 else 1)
        m = torch.from_numpy(m).to(x.device)
        x = torch.movedim(torch.tensordot(m, x, dims=([1], [a])), 0, a).contiguous()
    return x
