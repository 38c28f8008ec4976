"""The work that a user of this library has it do, as cases that can be timed and compared.

A case is a dict of plain values.  ``listed()`` gives the fixed ones, ``draw(rng)`` one more of the same ranges,
``prepare(case, seed)`` what a program holds before the call, ``run(state)`` one pass through the public entry points,
``work(case)`` the bytes and operations that pass cannot do without, ``tolerance(case)`` how close another correct
implementation comes.

Kinds of pass:

* ``linear``  one layer, one ``rabit_linear`` call, the output allocated by the call (the ordinary eager use);
* ``step``    the seven projections of one decoder layer, eager: q|k|v and gate|up as groups, o and down alone;
* ``token``   the same for a stack of decoder layers, captured once in a CUDA graph and replayed per token;
* ``host``    the decoder layer of ``step`` through the host-buffer form: pinned activations in, pinned results out, with
              the synchronisation that has to come before the results are read;
* ``derive``  loading a layer: sign planes derived from an fp32 weight on the device and packed;
* ``pack``    loading a layer: canonical sign planes in host memory packed and uploaded.

Layers are derived on the device from W ~ N(0, 0.02^2) with h ~ U(0.5, 1.5), g_1 ~ U(0.01, 0.03), g_k = g_{k-1} U(0.2, 0.5),
which makes every sign +-1 with probability one half; activations are N(0, 1) in fp16.
"""
import math

import numpy as np
import torch

import paper_2602_05367_b200 as rabit

DEVICE = "cuda:0"


def listed():
    return [
        # 8B-shaped k or v projection, one token: the smallest call, where latency counts
        {"name": "linear_kv_1024x4096_b1", "kind": "linear", "K": 2, "M": 1024, "N": 4096, "batch": 1},
        # one 7B-shaped decoder layer, one token, eager
        {"name": "step_7b_b1", "kind": "step", "K": 2, "d": 4096, "kv": 4096, "ffn": 11008, "batch": 1},
        # one token through the 32 layers of a 7B-shaped decoder: weights come from HBM, launches from a graph
        {"name": "token_7b_b1", "kind": "token", "K": 2, "layers": 32, "d": 4096, "kv": 4096, "ffn": 11008, "batch": 1},
        # sixteen sequences decoded together, 8B shapes
        {"name": "token_8b_b16", "kind": "token", "K": 2, "layers": 4, "d": 4096, "kv": 1024, "ffn": 14336, "batch": 16},
        # a decoder layer whose activations live in host memory
        {"name": "host_7b_b1", "kind": "host", "K": 2, "d": 4096, "kv": 4096, "ffn": 11008, "batch": 1},
        # 70B-shaped gate projection, two sequences
        {"name": "linear_28672x8192_b2", "kind": "linear", "K": 2, "M": 28672, "N": 8192, "batch": 2},
        # 8B-shaped down projection, five draft tokens verified at once
        {"name": "linear_4096x14336_b5", "kind": "linear", "K": 2, "M": 4096, "N": 14336, "batch": 5},
        # 8B-shaped gate projection, a server's decode batch
        {"name": "linear_14336x4096_b48", "kind": "linear", "K": 2, "M": 14336, "N": 4096, "batch": 48},
        # three paths, 13B-sized input, a row count that is no multiple of a tile, a short prompt
        {"name": "linear_5000x13824_k3_b200", "kind": "linear", "K": 3, "M": 5000, "N": 13824, "batch": 200},
        # 70B-shaped gate projection, prefill
        {"name": "linear_28672x8192_b512", "kind": "linear", "K": 2, "M": 28672, "N": 8192, "batch": 512},
        # load time: a 7B-shaped gate projection from its fp32 weight
        {"name": "derive_11008x4096", "kind": "derive", "K": 2, "M": 11008, "N": 4096},
        # load time: a 7B-shaped q projection from sign planes in host memory
        {"name": "pack_4096x4096", "kind": "pack", "K": 2, "M": 4096, "N": 4096},
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _paths(rng):
    return rng.choice((1, 2, 2, 2, 3))


def draw(rng):
    costs = [(c["kind"], work(c)) for c in listed()]
    kind = rng.choice(("linear",) * 12 + ("step", "step", "token", "token", "host", "derive", "derive", "pack"))
    while True:
        K = _paths(rng)
        M, N = _log_int(rng, 256, 28672), 32 * _log_int(rng, 16, 896)
        d = 128 * _log_int(rng, 8, 64)
        block = {"K": K, "d": d, "kv": d // rng.choice((1, 4, 8)), "ffn": 32 * int(d * rng.uniform(2.5, 3.6) / 32)}
        if kind == "linear":
            lo, hi = rng.choice(((1, 1), (1, 2), (3, 16), (3, 16), (17, 128), (17, 128), (129, 4096), (129, 4096)))
            case = {"kind": kind, "K": K, "M": M, "N": N, "batch": _log_int(rng, lo, hi)}
        elif kind == "step":
            case = dict(block, kind=kind, batch=rng.choice((1, 1, 2, 3, 4, 7, 8, 13, 16)))
        elif kind == "token":
            case = dict(block, kind=kind, layers=rng.randint(2, 8), batch=rng.choice((1, 1, 2, 4, 5, 8, 11, 16)))
        elif kind == "host":
            case = dict(block, kind=kind, batch=rng.choice((1, 1, 2, 4)))
        else:
            case = {"kind": kind, "K": K, "M": M, "N": N}
        w = work(case)
        if w["bytes"] <= max(c["bytes"] for k, c in costs if k == kind) and w["flops"] <= max(c["flops"] for _, c in costs):
            return case


# ---- making the inputs -----------------------------------------------------------------------------------

def _scales(rng, K, M, N):
    h = rng.uniform(0.5, 1.5, (K, N)).astype(np.float16)
    g = np.empty((K, M), dtype=np.float16)
    g[0] = rng.uniform(0.01, 0.03, M)
    for k in range(1, K):
        g[k] = g[k - 1].astype(np.float64) * rng.uniform(0.2, 0.5, M)
    return g, h


def _weight(gen, M, N):
    return torch.randn((M, N), generator=gen, dtype=torch.float32, device=DEVICE).mul_(0.02)


def _layer(gen, rng, K, M, N):
    g, h = _scales(rng, K, M, N)
    return rabit.rabit_derive_pack(_weight(gen, M, N), g, h)


def _x(gen, batch, N):
    return torch.randn((batch, N), generator=gen, dtype=torch.float32, device=DEVICE).to(torch.float16)


def _decoder_shapes(case):
    """(name, M, N, input) of the seven projections, in the order they are called."""
    d, kv, f = case["d"], case["kv"], case["ffn"]
    return [("q", d, d, "attn"), ("k", kv, d, "attn"), ("v", kv, d, "attn"), ("o", d, d, "mix"),
            ("gate", f, d, "mlp"), ("up", f, d, "mlp"), ("down", d, f, "act")]


GROUPS = ((0, 1, 2), (3,), (4, 5), (6,))        # the projections that share an input go through one call


def prepare(case, seed):
    gen = torch.Generator(device=DEVICE).manual_seed(seed)
    rng = np.random.default_rng(seed)
    kind, K = case["kind"], case["K"]
    if kind == "linear":
        return {"kind": kind, "layer": _layer(gen, rng, K, case["M"], case["N"]), "x": _x(gen, case["batch"], case["N"])}
    if kind == "derive":
        g, h = _scales(rng, K, case["M"], case["N"])
        return {"kind": kind, "W": _weight(gen, case["M"], case["N"]), "g": g, "h": h}
    if kind == "pack":
        g, h = _scales(rng, K, case["M"], case["N"])
        planes = rng.integers(0, 1 << 32, (K, case["M"], case["N"] // 32), dtype=np.uint32)
        return {"kind": kind, "planes": planes, "g": g, "h": h}

    shapes, batch = _decoder_shapes(case), case["batch"]
    x = {name: _x(gen, batch, n) for name, n in (("attn", case["d"]), ("mix", case["d"]), ("mlp", case["d"]), ("act", case["ffn"]))}
    blocks = [[_layer(gen, rng, K, M, N) for _, M, N, _ in shapes] for _ in range(case.get("layers", 1))]
    if kind == "host":
        x = {name: t.cpu().pin_memory() for name, t in x.items()}
        y = [torch.zeros((batch, M), dtype=torch.float16).pin_memory() for _, M, _, _ in shapes]
        calls = [rabit.PreparedGroupHost([blocks[0][i] for i in grp], [x[shapes[i][3]] for i in grp], [y[i] for i in grp]) for grp in GROUPS]
        return {"kind": kind, "calls": calls, "y": y}
    y = [torch.zeros((len(blocks), batch, M), dtype=torch.float16, device=DEVICE) for _, M, _, _ in shapes]
    state = {"kind": kind, "blocks": blocks, "x": [x[s[3]] for s in shapes], "y": y}
    if kind == "token":
        stream = torch.cuda.Stream()
        stream.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(stream):
            _decode(state)                       # once outside the capture
            stream.synchronize()
            state["graph"] = torch.cuda.CUDAGraph()
            with torch.cuda.graph(state["graph"], stream=stream):
                _decode(state)
        torch.cuda.current_stream().wait_stream(stream)
    return state


# ---- one pass --------------------------------------------------------------------------------------------

def _decode(state):
    x, y = state["x"], state["y"]
    for l, block in enumerate(state["blocks"]):
        for grp in GROUPS:
            if len(grp) == 1:
                i = grp[0]
                rabit.rabit_linear(block[i], x[i], y[i][l])
            else:
                rabit.rabit_linear_group([block[i] for i in grp], [x[i] for i in grp], [y[i][l] for i in grp])


def run(state):
    kind = state["kind"]
    if kind == "linear":
        return rabit.rabit_linear(state["layer"], state["x"])
    if kind == "step":
        _decode(state)
        return state["y"]
    if kind == "token":
        state["graph"].replay()
        return state["y"]
    if kind == "host":
        for call in state["calls"]:
            call()
        torch.cuda.current_stream().synchronize()
        return state["y"]
    if kind == "derive":
        return rabit.rabit_derive_pack(state["W"], state["g"], state["h"]).dev_buf
    return rabit.rabit_pack(state["planes"], state["g"], state["h"]).dev_buf


# ---- what a pass cannot do without, and how close results come -------------------------------------------

def _linear_work(K, M, N, batch):
    return {"bytes": K * M * N / 8 + 2 * K * (M + N) + 2 * batch * (M + N), "flops": 2.0 * K * M * N * batch}


def work(case):
    kind, K = case["kind"], case["K"]
    if kind == "linear":
        return _linear_work(K, case["M"], case["N"], case["batch"])
    if kind == "derive":
        return {"bytes": 4.0 * case["M"] * case["N"] + rabit.packed_bytes(K, case["M"], case["N"]), "flops": 0.0}
    if kind == "pack":
        return {"bytes": K * case["M"] * case["N"] / 8 + rabit.packed_bytes(K, case["M"], case["N"]), "flops": 0.0}
    parts = [_linear_work(K, M, N, case["batch"]) for _, M, N, _ in _decoder_shapes(case)]
    return {k: case.get("layers", 1) * sum(p[k] for p in parts) for k in ("bytes", "flops")}


def tolerance(case):
    # packed images are bytes; outputs are fp16 of fp32-accurate sums: one rounding (2^-11 of the value at most), which two
    # correct summation orders may take to neighbouring values
    return "exact" if case["kind"] in ("derive", "pack") else {"rel": 5e-4, "max": 2e-3}
