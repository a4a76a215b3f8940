"""The work that a user of this framework has it do, as measurable cases.

A case is one pass through the public entry points (``protocol`` and
``decoder``; the C ABI's binding ``mosaic`` for the rotation), as a serving or
model-loading program calls them.  Every case has a ``kind``:

  pass     Init X and the online part of one secure linear call (prefill)
  online   the online part alone, from masks drawn ahead (decode); with
           ``graph`` the calls of one token step are one CUDA graph, as a
           serving loop keeps it
  layer    a whole masked decoder layer (Init X, four secure linears, fp32 glue)
  load     Init W: the public chains of a width and one masked weight matrix
  check    Freivalds' check of a server answer
  rotate   the random Hadamard rotation of a batch of rows

Activations are N(0, 1) with a few outlier channels, weights N(0, 0.02), the
structure of transformer projections; keys, pass ids and inputs come from the
seed alone.  Sizes are those of the 7B and 70B projections and of the decode
sweep in ``workloads.py``, and generic odd ones.
"""
from __future__ import annotations

import math
from types import SimpleNamespace

import numpy as np
import torch
import torch.nn.functional as F

from paper_2607_29221_gb300 import decoder as D
from paper_2607_29221_gb300 import mosaic as M
from paper_2607_29221_gb300 import protocol as PR

RANKS, WEIGHTS = (1536, 1024, 652), (0, 80, 80)     # Example 3.1 parameters
SUM_R = sum(RANKS)

# (m, n) of the secure linears of one 70B decode step: QKV, O, gate+up, down.
DECODE_70B = ((10240, 8192), (8192, 8192), (57344, 8192), (8192, 28672))


def listed():
    return [
        # A small linear on a few tokens: launches and host work are all of it.
        {"name": "pass_64x256x128", "kind": "pass", "l": 64, "m": 128, "n": 256, "nested": True, "bias": True},
        # Prefill of a 512-token batch through the 7B attention projection.
        {"name": "pass_attn_7b_512", "kind": "pass", "l": 512, "m": 4096, "n": 4096, "nested": True, "bias": True},
        # The same with the LWE-only activation mask (act_nested = 0), the variant the paper deploys.
        {"name": "pass_lwe_only_512", "kind": "pass", "l": 512, "m": 4096, "n": 4096, "nested": False, "bias": True},
        # A ragged batch through a matrix of odd width and height (an output head, an adapter).
        {"name": "pass_odd_301x3001x5003", "kind": "pass", "l": 301, "m": 5003, "n": 3001, "nested": True,
         "bias": False},
        # One generated token: the four secure linears of a 70B layer, masks drawn ahead, one CUDA graph.
        {"name": "decode_70b_1", "kind": "online", "l": 1, "m": 0, "n": 0, "graph": True},
        # A decode batch of 8 through the 70B output projection, called without a graph.
        {"name": "decode_o_70b_8", "kind": "online", "l": 8, "m": 8192, "n": 8192, "graph": False},
        # A decode batch of 32: the four secure linears of a 70B layer as one CUDA graph.
        {"name": "decode_70b_32", "kind": "online", "l": 32, "m": 0, "n": 0, "graph": True},
        # A large decode batch through the 70B fused QKV projection.
        {"name": "decode_qkv_70b_128", "kind": "online", "l": 128, "m": 10240, "n": 8192, "graph": False},
        # Loading a model: the public chains of the width and Init W of the 7B attention projection.
        {"name": "load_attn_7b", "kind": "load", "m": 4096, "n": 4096},
        # Checking a 512-token answer of the 70B output projection with 4 vectors.
        {"name": "check_o_70b_512", "kind": "check", "l": 512, "m": 8192, "n": 8192, "k": 4},
        # The rotation of a 2048-token batch of the 7B FFN's inner width (padded to 16384).
        {"name": "rotate_2048x14336", "kind": "rotate", "l": 2048, "n": 14336},
        # The whole 70B decoder layer, prefill of 2048 tokens.
        {"name": "layer_70b_2048", "kind": "layer", "l": 2048, "hidden": 8192, "heads": 64, "kv": 8, "ffn": 28672},
    ]


def _log(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _size(rng, lo, hi):
    """Half of the sizes a multiple of 64 (model widths), the others as they fall."""
    v = _log(rng, lo, hi)
    return max(64, v // 64 * 64) if rng.random() < 0.5 else v


def draw(rng):
    kind = rng.choice(["pass", "pass", "pass", "online", "online", "online", "layer", "load", "check", "rotate"])
    if kind == "pass":
        return {"kind": kind, "l": _log(rng, 1, 2048), "m": _size(rng, 128, 16384), "n": _size(rng, 256, 16384),
                "nested": rng.random() < 0.75, "bias": rng.random() < 0.5}
    if kind == "online":
        return {"kind": kind, "l": _log(rng, 1, 256), "m": _size(rng, 1024, 57344), "n": _size(rng, 1024, 16384),
                "graph": rng.random() < 0.5}
    if kind == "layer":
        kv = rng.choice([2, 4, 8])
        heads = kv * rng.choice([1, 4, 8])
        return {"kind": kind, "l": _log(rng, 65, 2048), "hidden": heads * 128, "heads": heads, "kv": kv,
                "ffn": 128 * _log(rng, heads * 2, heads * 4)}
    if kind == "load":
        return {"kind": kind, "m": _size(rng, 256, 16384), "n": _size(rng, 256, 16384)}
    if kind == "check":
        return {"kind": kind, "l": _log(rng, 1, 2048), "m": _size(rng, 256, 16384), "n": _size(rng, 256, 16384),
                "k": rng.randint(1, 16)}
    return {"kind": kind, "l": _log(rng, 16, 8192), "n": _size(rng, 256, 32768)}


# ---------------------------------------------------------------------------
def _pairs(case):
    """(m, n) of the secure linears of a pass or online case."""
    return ((case["m"], case["n"]),) if case["m"] else DECODE_70B


def _layer_pairs(case):
    h, f = case["hidden"], case["ffn"]
    return (((case["heads"] + 2 * case["kv"]) * 128, h), (h, case["heads"] * 128), (2 * f, h), (h, f))


def _gen(seed, salt=0):
    g = torch.Generator(device="cuda")
    g.manual_seed(1_000_003 * seed + salt)
    return g


def _activations(g, l, n):
    x = torch.randn(l, n, generator=g, device="cuda")
    x[:, torch.randint(0, n, (4,), generator=g, device="cuda")] *= 20.0
    return x


def _weights(g, m, n):
    return torch.randn(m, n, generator=g, device="cuda") * 0.02


def _protocol(seed, nested=True):
    key = np.random.Generator(np.random.PCG64(seed)).integers(0, 1 << 32, 8, dtype=np.uint32)
    return PR.Protocol(key, M.default_params(act_nested=1 if nested else 0))


def _inputs(case, seed):
    """The float inputs of a case: what both `prepare` and `exact` start from."""
    g = _gen(seed)
    kind = case["kind"]
    if kind in ("pass", "online"):
        return [(_weights(g, m, n), _activations(g, case["l"], n),
                 torch.randn(m, generator=g, device="cuda") * 0.02 if case.get("bias", False) else None)
                for m, n in _pairs(case)]
    if kind == "layer":
        x = _activations(g, case["l"], case["hidden"])
        return x, [_weights(g, m, n) for m, n in _layer_pairs(case)]
    if kind in ("load", "check"):
        return _weights(g, case["m"], case["n"])
    n_pad = PR.pad_width(case["n"])
    return (_activations(g, case["l"], case["n"]),
            torch.randint(-(1 << 31), 1 << 31, (n_pad // 32,), generator=g, device="cuda", dtype=torch.int64)
            .to(torch.int32))


def prepare(case, seed):
    kind, l = case["kind"], case.get("l", 0)
    s = SimpleNamespace(case=case, pass_id=1 + 1000 * (seed % 100_000))
    if kind in ("pass", "online"):
        proto = _protocol(seed, case.get("nested", True))
        chains, s.lins, s.xs = {}, [], []
        for i, (W, x, b) in enumerate(_inputs(case, seed)):
            n_pad = PR.pad_width(W.shape[1])
            if n_pad not in chains:
                chains[n_pad] = PR.Chains(proto, n_pad)
            s.lins.append(PR.SecureLinear(proto, W, 1 + i, chains[n_pad], bias=b))
            s.xs.append(x)
        if kind == "online":
            s.masks = [lin.init_x(l, s.pass_id + i) for i, lin in enumerate(s.lins)]
            if case["graph"]:
                _online(s)                                   # sizes the workspace
                torch.cuda.synchronize()
                s.graph = torch.cuda.CUDAGraph()
                with torch.cuda.graph(s.graph):
                    s.Y = _online(s)
                torch.cuda.synchronize()
    elif kind == "layer":
        s.x, (qkv, o, gu, down) = _inputs(case, seed)
        shape = D.LayerShape(hidden=case["hidden"], n_heads=case["heads"], n_kv=case["kv"], ffn=case["ffn"])
        w = SimpleNamespace(s=shape, Wqkv=qkv, Wo=o, Wgu=gu, Wdown=down)
        s.layer = D.SecureDecoderLayer(_protocol(seed), w)
        s.layer.alloc(l)
        s.masks = [PR.PassMask(0, l, torch.empty(l, lin.n_pad, dtype=torch.int32, device="cuda"),
                               torch.empty(l, lin.m, dtype=torch.int32, device="cuda"))
                   for lin in s.layer.linears()]
    elif kind == "load":
        s.seed, s.W, s.n_pad = seed, _inputs(case, seed), PR.pad_width(case["n"])
        s.proto = _protocol(seed)
    elif kind == "check":
        W = _inputs(case, seed)
        s.lin = PR.SecureLinear(_protocol(seed), W, 1, PR.Chains(_protocol(seed), PR.pad_width(case["n"])))
        s.lin.freivalds_setup(case["k"])
        Xp, _, Xpl = s.lin.mask_input(_activations(_gen(seed, 1), l, case["n"]), s.lin.init_x(l, s.pass_id))
        s.Xp, s.Z = Xp, s.lin.server(Xp, Xpl)
        # A dishonest server: single entries of a few tokens' answers are off.
        at = torch.randint(0, l * case["m"], (1 + l // 64,), generator=_gen(seed, 2), device="cuda")
        s.Z[at // case["m"], at % case["m"]] += 12345
    else:
        s.x, s.signs = _inputs(case, seed)
        s.y = torch.empty(l, PR.pad_width(case["n"]), device="cuda")
    return s


def _online(s):
    return [lin.forward(x, mp) for lin, x, mp in zip(s.lins, s.xs, s.masks)]


def run(s):
    case = s.case
    kind = case["kind"]
    if kind == "pass":
        lin = s.lins[0]
        mp = lin.init_x(case["l"], s.pass_id)
        return {"Ux": mp.Ux, "K": mp.K, "Y": lin.forward(s.xs[0], mp)}
    if kind == "online":
        if not case["graph"]:
            return {"Y": _online(s)}
        s.graph.replay()
        return {"Y": s.Y}
    if kind == "layer":
        return {"Y": s.layer.forward_pass(s.x, s.pass_id, s.masks),
                "Ux": [mp.Ux for mp in s.masks], "K": [mp.K for mp in s.masks]}
    if kind == "load":
        ch = PR.Chains(s.proto, s.n_pad)
        lin = PR.SecureLinear(s.proto, s.W, 1, ch)
        return {"P": ch.P, "C": ch.C, "CT": ch.CT, "signs": lin.sign_words, "s_w": lin.s_w, "L": lin.L,
                "S_idx": lin.S_idx, "S_val": lin.S_val, "Wp": lin.Wp, "Wp_planes": lin.Wp_planes, "J": lin.J}
    if kind == "check":
        bad, n_bad = s.lin.freivalds_check(s.Z, s.Xp)
        return {"bad": bad, "n_bad": n_bad}
    M.mosaic_hadamard(s.x, s.x.stride(0), s.y, case["l"], case["n"], s.y.shape[1], s.signs)
    return {"y": s.y}


# ---------------------------------------------------------------------------
def _linear_work(l, m, n, nested, init_x):
    """Bytes and operations of one secure linear call.  A ring multiply-add of
    the dense products is counted as the 10 exact digit products of 8 bits it
    takes on the tensor cores (20 operations), one of the sparse LPN terms as
    2.  The client keeps C, J, L, S; the server W' and P, 4 bytes each."""
    n_pad = PR.pad_width(n)
    sparse = sum(WEIGHTS)
    flops = 20 * l * (m + SUM_R) * n_pad + 20 * l * m * RANKS[-1] + 2 * l * m * sparse
    byts = 4 * (l * n + n_pad * (m + SUM_R) + m * RANKS[-1] + 2 * m * sparse + l * m)
    if init_x:
        rank, cols = (RANKS[-1], SUM_R) if nested else (RANKS[0], RANKS[0])
        flops += 20 * l * (n_pad + m) * rank + (2 * l * (n_pad + m) * sparse if nested else 0)
        byts += 4 * ((n_pad + m) * cols + l * (n_pad + m))
    else:
        byts += 4 * l * (n_pad + m)
    return byts, flops


def work(case):
    kind, l = case["kind"], case.get("l", 0)
    if kind in ("pass", "online"):
        parts = [_linear_work(l, m, n, case.get("nested", True), kind == "pass") for m, n in _pairs(case)]
    elif kind == "layer":
        parts = [_linear_work(l, m, n, True, True) for m, n in _layer_pairs(case)]
        parts.append((0, 2 * l * l * case["heads"] * 128))           # causal attention: half of 4 l^2 d per head
    elif kind == "load":
        m, n_pad = case["m"], PR.pad_width(case["n"])
        chain = sum(a * b for a, b in zip(RANKS[:-1], RANKS[1:])) * n_pad * 2
        flops = 20 * (chain + m * n_pad * (SUM_R + RANKS[-1])) + 2 * m * n_pad * sum(WEIGHTS)
        # W in; P, C, C^T, [W'; P] and its digit planes, J, L and S out.
        byts = 4 * (m * case["n"] + 3 * SUM_R * n_pad + 3 * (m + SUM_R) * n_pad + m * (SUM_R + RANKS[-1])
                    + 2 * m * sum(WEIGHTS))
        parts = [(byts, flops)]
    elif kind == "check":
        m, n_pad, k = case["m"], PR.pad_width(case["n"]), case["k"]
        parts = [(4 * ((l + k) * (m + n_pad) + l), 2 * k * l * (m + n_pad))]
    else:
        n_pad = PR.pad_width(case["n"])
        parts = [(4 * l * (case["n"] + n_pad), l * n_pad * (n_pad.bit_length() - 1))]
    return {"bytes": sum(p[0] for p in parts), "flops": sum(p[1] for p in parts)}


def tolerance(case):
    """Ring outputs are exact by definition, and the float steps of a secure
    linear have their order and roundings fixed by the API (fp32 butterflies in
    stage order, IEEE division, two products and an add in the decode).  The
    layer's softmax attention and norms have not: a change of their summation
    order moves a few quantised codes in every linear that follows.  Measured
    with the attention or the norms summed in another order: rel 0.0055 / max
    0.031 at hidden 8192, 0.0026 / 0.014 at 4096, 8e-6 / 8e-5 at 512 and 8e-7 /
    2e-5 at 256, where the update is small beside the residual; four times that."""
    if case["kind"] != "layer":
        return "exact"
    rel = min(0.022, 3.4e-5 * (case["hidden"] / 512) ** 2.8)
    return {"rel": rel, "max": min(0.12, 40 * rel)}


def _attention64(qkv, heads, kv):
    l, d = qkv.shape[0], 128
    out = torch.empty(l, heads * d, dtype=torch.float64, device="cuda")
    mask = torch.ones(l, l, dtype=torch.bool, device="cuda").tril()
    for h in range(heads):
        g = h // (heads // kv)
        q = qkv[:, h * d:(h + 1) * d]
        k = qkv[:, (heads + g) * d:(heads + g + 1) * d]
        v = qkv[:, (heads + kv + g) * d:(heads + kv + g + 1) * d]
        sc = (q @ k.T / math.sqrt(d)).masked_fill(~mask, -math.inf)
        out[:, h * d:(h + 1) * d] = torch.softmax(sc, 1) @ v
    return out


def _linear64(x, W, b=None):
    y = torch.cat([x @ w.double().T for w in W.split(4096)], 1)
    return y if b is None else y + b.double()


def exact(case, seed):
    """What the secure layers approximate, in 64 bits: the plain linear layer
    or decoder layer (the noise of the masks and the quantisation are the
    method's own error, about 0.5%), and the rotation itself.  Ring values and
    masks have no such value."""
    kind = case["kind"]
    if kind == "pass":
        W, x, b = _inputs(case, seed)[0]
        return {"Ux": None, "K": None, "Y": _linear64(x.double(), W, b)}
    if kind == "online":
        return {"Y": [_linear64(x.double(), W, b) for W, x, b in _inputs(case, seed)]}
    if kind == "layer":
        x, (qkv, o, gu, down) = _inputs(case, seed)
        x = x.double()

        def norm(v):
            return v / torch.sqrt((v * v).mean(1, keepdim=True) + 1e-5)

        x = x + _linear64(_attention64(_linear64(norm(x), qkv), case["heads"], case["kv"]), o)
        g, u = _linear64(norm(x), gu).split(case["ffn"], 1)
        return {"Y": x + _linear64(F.silu(g) * u, down), "Ux": None, "K": None}
    if kind == "rotate":
        x, signs = _inputs(case, seed)
        l, n = x.shape
        n_pad = PR.pad_width(n)
        y = F.pad(x.double(), (0, n_pad - n))
        bits = (signs.to(torch.int64)[:, None] >> torch.arange(32, device="cuda")) & 1
        y = y * (1.0 - 2.0 * bits.reshape(-1).double())
        h = 1
        while h < n_pad:
            y = y.reshape(l, n_pad // (2 * h), 2, h)
            y = torch.stack((y[:, :, 0] + y[:, :, 1], y[:, :, 0] - y[:, :, 1]), 2)
            h *= 2
        return {"y": y.reshape(l, n_pad) / math.sqrt(n_pad)}
    return None
