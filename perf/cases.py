"""Performance cases of the AWSRC library: what its users have it do, over the sizes they use.

A repair of a model goes encode -> select -> decode over the linear modules of its layers
(once per model and operating point); a served model is quantised once and then multiplied
token by token from the packed backbone. Each case is one public entry point on the modules
of one or a few decoder layers (or one matrix), with output and workspace buffers kept by the
caller between calls, as a program that walks a model's layers keeps them.

Inputs follow the recipes of the repository's synthetic workloads (Qwen2.5 projection shapes,
N(0, 0.02^2) weights with Student-t outlier channels, lognormal activation moments, an
RTN-INT4 g128 backbone, lognormal Fisher diagonals) and are made here with plain torch, so
that they do not depend on the code that is measured.
"""
from __future__ import annotations

import math
import struct

import numpy as np
import torch

import paper_2608_23144_gb300 as aw

DEV = "cuda"
DTYPES = {"bf16": torch.bfloat16, "f32": torch.float32}


# ------------------------------------------------------------------ cases --

def _case(op, shape, hidden, inter=0, kv=0, layers=1, dtype="bf16", C=64, P=4, b=4, S=4096, variant="U", scale="pow2",
          rate=0.162, **kw):
    """shape: "layer" (7 modules), "attn" (q, k, v, o), "mlp" (gate, up, down) or "single"
    (one inter x hidden matrix)."""
    return dict(op=op, shape=shape, hidden=hidden, inter=inter, kv=kv, layers=layers, dtype=dtype, C=C, P=P, b=b, S=S,
                variant=variant, scale=scale, rate=rate, **kw)


def listed():
    q3 = dict(hidden=2048, inter=11008, kv=256)
    q7 = dict(hidden=3584, inter=18944, kv=512)
    cases = {
        # the small synthetic matrix: one call on one 256 x 512 projection, where launches count
        "encode_u_256x512": _case("encode", "single", 512, 256, dtype="f32", S=256, scale="fp16"),
        # the benchmark's step: the seed search of one whole 3B-shaped layer
        "encode_u_layer": _case("encode", "layer", **q3),
        # the Fisher-weighted search on a 7B-shaped attention block
        "encode_pf_attn": _case("encode", "attn", variant="PF", **q7),
        # the paper's two operating points on the MLP projections (its own scope)
        "encode_u_c128_mlp": _case("encode", "mlp", C=128, P=2, S=2, **q3),
        "encode_pf_c16_mlp": _case("encode", "mlp", C=16, S=16, variant="PF", **q3),
        # allocation and serialisation of one layer under U
        "select_u_layer": _case("select", "layer", **q3),
        # one global ranking of four 7B-shaped layers, cut at four rates
        "select_pf_4_layers": _case("select", "layer", layers=4, variant="PF", rate=0.25, **q7),
        # loading a repaired layer: dense decode of the whole stream
        "decode_u_layer": _case("decode", "layer", mode="dense", out="bf16", **q3),
        # the longest progressive prefix of a larger layer
        "decode_pf_layer": _case("decode", "layer", variant="PF", rate=0.25, mode="dense", out="bf16", **q7),
        # the backbone of a layer, scales double quantised
        "rtn_sdq_layer": _case("rtn", "layer", sdq=True, **q3),
        # one token through a layer's projections, and eight (a small batch of requests)
        "gemv_layer_m1": _case("gemv", "layer", sdq=True, M=1, **q3),
        "gemv_layer_m8": _case("gemv", "layer", sdq=True, M=8, **q3),
    }
    return [dict(c, name=n) for n, c in cases.items()]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    while True:
        op = rng.choice(["encode"] * 4 + ["select", "decode", "decode", "rtn", "gemv", "gemv"])
        shape = rng.choice(["layer", "attn", "mlp", "single", "single"])
        hidden = 128 * max(2, round(_log(rng, 2, 40)))
        c = dict(shape=shape, hidden=hidden, inter=128 * round(hidden * rng.uniform(2.5, 5.5) / 128),
                 kv=128 * rng.randint(1, max(1, hidden // 512)), dtype=rng.choice(["bf16", "bf16", "bf16", "f32"]))
        if shape == "single":  # any number of rows, odd ones among them
            c["inter"] = round(_log(rng, 16, 20000))
        variant = rng.choice(["U", "U", "PF"])
        if rng.random() < 0.6:
            codec = dict(C=64, P=4, S=rng.choice([4096, round(_log(rng, 64, 4096))]))
        else:
            codec = dict(C=rng.choice([16, 32, 128]), P=rng.choice([2, 4]), S=rng.choice([2, 4, 16, round(_log(rng, 2, 64))]))
        codec.update(variant=variant, scale=rng.choice(["pow2", "pow2", "pow2", "fp16"]),
                     rate=rng.choice([0.05, 0.10, 0.162, 0.25]))
        more = {}
        if op == "select":
            more["layers"] = rng.randint(1, 4)
        elif op == "decode":
            mode = rng.choice(["dense", "dense", "inplace"])
            more = dict(mode=mode, out=rng.choice(["bf16", "bf16", "f32"]) if mode == "dense" else c["dtype"])
        elif op == "rtn":
            more["sdq"] = rng.random() < 0.5
        elif op == "gemv":
            more = dict(sdq=rng.random() < 0.5, M=rng.randint(1, 8), layers=1)
        case = _case(op, **c, **codec, **more)
        if _us(case) < 8500 and _stream_room(case):
            return case


def _shapes(case):
    h, i, kv = case["hidden"], case["inter"], case["kv"]
    attn = [(h, h), (kv, h), (kv, h), (h, h)]
    mlp = [(i, h), (i, h), (h, i)]
    one = {"layer": attn + mlp, "attn": attn, "mlp": mlp, "single": [(i, h)]}[case["shape"]]
    return one * case["layers"]


def _weights(case):
    return sum(r * c for r, c in _shapes(case))


def _us(case):
    """A rough time of one pass, to keep drawn cases below the largest listed one."""
    N, T = _weights(case), _weights(case) / case["C"]
    if case["op"] == "encode":
        per = 1.8e-6 if case["variant"] == "U" else 4.9e-6
        if (case["C"], case["P"]) != (64, 4):
            per = 1e-4
        return N * 5e-6 + T * case["S"] * per
    if case["op"] == "select":
        return T * 3e-4
    return N * (4e-5 if case["op"] == "gemv" else 2.5e-5)


def _stream_room(case):
    """The byte budget has to hold the stream's header and a few records."""
    return _weights(case) * case["rate"] / 8 > 40 + 8 * len(_shapes(case)) + 16 * 64


def work(case):
    """Each input read once, each output written once; the search's flops are the Eq. 3
    correlations (and, for P_F, the Gram's), 2 C per sum."""
    shapes, C, P = _shapes(case), case["C"], case["P"]
    N = _weights(case)
    T = N // C
    wb = 2 if case["dtype"] == "bf16" else 4
    cols = sum(c for _, c in shapes)
    K, L, h = _stream_size(case)
    if case["op"] == "encode":
        pf = case["variant"] == "PF"
        sums = P + (P * (P - 1) // 2 if pf else 0)
        return {"bytes": N * (2 * wb + (4 if pf else 0)) + 4 * cols + 16 * T, "flops": 2.0 * C * sums * T * case["S"]}
    if case["op"] == "select":  # every gain once, the kept candidates, the stream
        return {"bytes": 4 * T + 16 * K + h + K * L, "flops": 0}
    if case["op"] == "decode":
        ob = 2 if case["out"] == "bf16" else 4
        n = N if case["mode"] == "dense" else K * C
        return {"bytes": n * (wb + ob) + h + K * L, "flops": 2.0 * P * C * K}
    meta = N // 128 + 8 * sum(-(-r * c // 128 // 256) for r, c in shapes) if case["sdq"] else N // 64
    if case["op"] == "rtn":
        return {"bytes": N * wb + N // 2 + N // 64 + (meta if case["sdq"] else 0) + N * wb, "flops": 2.0 * N}
    M = case["M"]
    return {"bytes": N // 2 + meta + h + K * L + 4 * M * sum(r + c for r, c in shapes), "flops": 2.0 * M * N}


# ----------------------------------------------------------------- inputs --

def _params(case):
    return aw.params(C=case["C"], P=case["P"], b=case["b"], S=case["S"], b_e=8 if case["scale"] == "pow2" else 16,
                     scale_mode=aw.SCALE_POW2 if case["scale"] == "pow2" else aw.SCALE_FP16,
                     variant=aw.VARIANT_U if case["variant"] == "U" else aw.VARIANT_PF)


def _bits(n):
    return max(0, (n - 1).bit_length())


def _stream_size(case):
    """(records, bytes per record, header bytes) of the stream at the case's rate."""
    shapes = _shapes(case)
    N, T = _weights(case), _weights(case) // case["C"]
    b_e = 8 if case["scale"] == "pow2" else 16
    L = (_bits(T) + _bits(case["S"]) + b_e + case["P"] * case["b"] + 7) // 8
    h = 40 + 8 * len(shapes)
    B = int(math.floor(case["rate"] * N / 8.0))
    if case["variant"] == "PF":
        return min((B - h) // L, T), L, h
    return sum(_quotas(case, B - h, L)), L, h


def _quotas(case, room, L):
    N = _weights(case)
    return [min(room * r * c // N // L, r * c // case["C"]) for r, c in _shapes(case)]


def _weight(rows, cols, g):
    W = torch.randn(rows, cols, generator=g, device=DEV) * 0.02
    n = max(1, round(0.01 * cols))
    oc = torch.randperm(cols, generator=g, device=DEV)[:n]
    chi = (torch.randn(rows, n, 4, generator=g, device=DEV) ** 2).sum(-1)
    W[:, oc] = 0.16 * torch.randn(rows, n, generator=g, device=DEV) / torch.sqrt(chi / 4)
    return W


def _act(cols, g):
    """Second moments of 1024 tokens of a channel of standard deviation s: s^2 chi^2_1024 / 1024."""
    s2 = torch.exp(2 * torch.randn(cols, generator=g, device=DEV))
    return s2 * (1 + math.sqrt(2 / 1024) * torch.randn(cols, generator=g, device=DEV)).clamp_min(0.5)


def _rtn(W, sdq, dt=torch.float32):
    """RTN-INT4, groups of 128 inputs: codes, binary16 scales, (SDQ codes and constants), q * scale."""
    rows, cols = W.shape
    w = W.to(dt).reshape(-1, 128)
    s = (w.abs().amax(1) / 7).half().to(dt)
    q = torch.clamp(torch.round(w / torch.where(s > 0, s, torch.ones_like(s))[:, None]), -8, 7)
    q = torch.where(s[:, None] > 0, q, torch.zeros_like(q))
    n = q.to(torch.int32).reshape(-1, 2) & 15
    out = {"codes": (n[:, 0] | (n[:, 1] << 4)).to(torch.uint8), "scales": s.half().view(torch.int16)}
    if sdq:
        G = s.numel()
        nb = -(-G // 256)
        blk = torch.arange(G, device=s.device) // 256
        cnt = torch.zeros(nb, dtype=torch.float64, device=s.device).index_add_(0, blk, torch.ones(G, dtype=torch.float64, device=s.device))
        mu = (torch.zeros(nb, dtype=torch.float64, device=s.device).index_add_(0, blk, s.double()) / cnt).to(dt)
        dev = s - mu[blk]
        step = torch.zeros(nb, dtype=dt, device=s.device).scatter_reduce_(0, blk, dev.abs(), "amax") / 127
        c = torch.clamp(torch.round(dev / torch.where(step > 0, step, torch.ones_like(step))[blk]), -127, 127)
        out["sdq_codes"] = c.to(torch.int8)
        out["sdq_consts"] = torch.stack([mu, step], 1).reshape(-1).contiguous()
        s = mu[blk] + c * step[blk]
    out["W0"] = (q * s[:, None]).reshape(rows, cols)
    return out


def _energy(rows, cols, C, g, act, fisher):
    """Weighted error of every tile of an RTN residual (what gains are a share of)."""
    n = rows * (cols // C)
    out = torch.empty(n, device=DEV)
    step = max(1, (1 << 26) // cols)
    for r0 in range(0, rows, step):
        r = min(step, rows - r0)
        d = act * (0.006 * (torch.rand(r, cols, generator=g, device=DEV) - 0.5)) ** 2
        if fisher:
            d = d * (0.5 + 0.5 * torch.exp(1.5 * torch.randn(r, cols, generator=g, device=DEV)))
        out[r0 * (cols // C):(r0 + r) * (cols // C)] = d.reshape(-1, C).sum(1)
    return out


def _records(case, n, g):
    """Seeds, scale fields and codes of n records: codes are a Gaussian fit scaled to its largest."""
    P, qmax = case["P"], 2 ** (case["b"] - 1) - 1
    seed = torch.randint(0, case["S"], (n,), generator=g, device=DEV)
    a = torch.randn(n, P, generator=g, device=DEV)
    top = a.abs().amax(1, keepdim=True)
    code = torch.round(a / top * (qmax * (0.5 + 0.5 * torch.rand(n, 1, generator=g, device=DEV)))).to(torch.int64)
    if case["scale"] == "pow2":
        scale = torch.randint(-11, -7, (n,), generator=g, device=DEV)
    else:
        scale = (0.0005 * torch.exp(0.5 * torch.randn(n, generator=g, device=DEV))).half().view(torch.int16).long()
    return seed, scale, code


def _gains(case, g):
    """A gain per tile, module by module: a tenth to a third of the tile's weighted error, and
    nothing to gain (or no valid fit) on a few."""
    out = []
    for rows, cols in _shapes(case):
        e = _energy(rows, cols, case["C"], g, _act(cols, g), case["variant"] == "PF")
        e *= 0.1 + 0.2 * torch.rand(e.numel(), generator=g, device=DEV)
        u = torch.rand(e.numel(), generator=g, device=DEV)
        e = torch.where(u < 0.002, -e, e)
        out.append(torch.where(u < 0.001, torch.full_like(e, -math.inf), e))
    return out


def _candidates(case, g):
    gain = torch.cat(_gains(case, g))
    seed, scale, code = _records(case, gain.numel(), g)
    out = torch.zeros(gain.numel(), 16, dtype=torch.uint8, device=DEV)
    out[:, 0:4] = gain.view(torch.uint8).reshape(-1, 4)
    out[:, 4:6] = seed.to(torch.int32).to(torch.int16).view(torch.uint8).reshape(-1, 2)
    out[:, 6:8] = scale.to(torch.int16).view(torch.uint8).reshape(-1, 2)
    out[:, 8:8 + case["P"]] = code.to(torch.int8).view(torch.uint8)
    return out


def _stream(case, g):
    """A stream as the selection writes it: (device bytes, tile, seed, scale, code of its records)."""
    shapes, C = _shapes(case), case["C"]
    K, L, h = _stream_size(case)
    gains = _gains(case, g)
    if case["variant"] == "U":
        quota, off, parts = _quotas(case, int(math.floor(case["rate"] * _weights(case) / 8.0)) - h, L), 0, []
        for gm, k in zip(gains, quota):
            k = min(k, int((gm > 0).sum()))
            parts.append(off + torch.argsort(gm, descending=True)[:k])
            off += gm.numel()
        tile = torch.cat(parts)
    else:
        gain = torch.cat(gains)
        tile = torch.argsort(gain, descending=True)[:min(K, int((gain > 0).sum()))]
    K = tile.numel()
    seed, scale, code = _records(case, K, g)
    T = sum(r * c for r, c in shapes) // C
    b_e = 8 if case["scale"] == "pow2" else 16
    bits = torch.zeros(K, 8 * L, dtype=torch.uint8, device=DEV)
    pos = 0
    for v, n in [(tile, _bits(T)), (seed, _bits(case["S"])), (scale, b_e)] + [(code[:, p], case["b"]) for p in range(case["P"])]:
        for i in range(n):
            bits[:, pos + i] = ((v >> i) & 1).to(torch.uint8)
        pos += n
    body = (bits.reshape(K, L, 8) << torch.arange(8, dtype=torch.uint8, device=DEV)).sum(-1).to(torch.uint8)
    head = struct.pack("<IHBBHBBBbBBIIQQ", 0x52535741, 1, int(case["variant"] == "PF"), int(case["scale"] != "pow2"), C,
                       case["P"], case["b"], b_e, 0, 1, 0, case["S"], len(shapes), 0, K)
    off = 0
    for r, c in shapes:
        n = r * (c // C)
        head += struct.pack("<II", n, int(((tile >= off) & (tile < off + n)).sum()))
        off += n
    head = torch.from_numpy(np.frombuffer(head, dtype=np.uint8).copy()).to(DEV)
    return torch.cat([head, body.reshape(-1)]), tile, seed, scale, code


def _modules(case, g, W=True):
    """The dicts the entry points take, one per module."""
    out = []
    for rows, cols in _shapes(case):
        w = _weight(rows, cols, g).to(DTYPES[case["dtype"]])
        m = {"W0": _rtn(w, False)["W0"].to(w.dtype), "act": _act(cols, g)}
        if W:
            m["W"] = w
        if case["variant"] == "PF" and W:
            m["fisher"] = torch.exp(1.5 * torch.randn(rows, cols, generator=g, device=DEV))
            m["w_act"] = 0.5 / float(m["act"].mean())
            m["w_fisher"] = 0.5 / float(m["fisher"].mean())
        out.append(m)
    return out


def prepare(case, seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    st = {"case": case, "prm": _params(case), "ws": None}
    if case["op"] == "encode":
        st["mods"] = _modules(case, g)
        st["out"] = torch.empty(_weights(case) // case["C"], 16, dtype=torch.uint8, device=DEV)
    elif case["op"] == "select":
        # the selection reads shapes and candidates only: one small buffer stands for the weights
        # of every module (nothing but its shape is used)
        st["mods"] = [{"W0": torch.empty(r, c, dtype=torch.bfloat16, device=DEV)} for r, c in _shapes(case)]
        st["cands"] = _candidates(case, g)
        r = case["rate"]
        st["rates"] = [r] if case["variant"] == "U" else sorted({r * f for f in (0.2, 0.4, 0.648, 1.0)})
        st["buf"] = {}
    elif case["op"] == "decode":
        st["mods"] = _modules(case, g, W=False)
        st["records"] = _stream(case, g)
        st["out"] = [m["W0"].to(DTYPES[case["out"]], copy=True) for m in st["mods"]]  # in place: holds W0
    elif case["op"] == "rtn":
        st["Ws"] = [_weight(r, c, g).to(DTYPES[case["dtype"]]) for r, c in _shapes(case)]
        st["out"] = None
    else:
        st["shapes"] = _shapes(case)
        st["packed"] = [_rtn(_weight(r, c, g).to(torch.bfloat16), case["sdq"]) for r, c in st["shapes"]]
        for p in st["packed"]:
            del p["W0"]
        st["records"] = _stream(case, g)
        st["sidecar"] = aw.awsrc_sidecar_prepare(st["prm"], st["shapes"], st["records"][0])
        # the modules that share an input (q, k, v; gate, up) share x
        xs = {}
        st["tasks"] = []
        for i, (r, c) in enumerate(st["shapes"]):
            key = (i // 7, {0: 0, 1: 0, 2: 0, 4: 1, 5: 1}.get(i % 7, 2 + i)) if case["shape"] == "layer" else i
            if key not in xs:
                xs[key] = torch.randn(case["M"], c, generator=g, device=DEV)
            st["tasks"].append((i, st["packed"][i], xs[key], torch.empty(case["M"], r, device=DEV)))
    return st


def run(st):
    op, prm = st["case"]["op"], st["prm"]
    if op == "encode":
        out = aw.awsrc_encode_tiles(prm, st["mods"], out=st["out"], workspace=st["ws"])
        st["ws"] = out._awsrc_workspace
        return out
    if op == "select":
        b = st["buf"]
        out, counts, nbytes = aw.awsrc_select_records(prm, st["mods"], st["cands"], st["rates"], workspace=st["ws"],
                                                      out=b.get("out"), counts=b.get("counts"), nbytes=b.get("nbytes"))
        st["ws"] = out._awsrc_workspace
        st["buf"] = dict(out=out, counts=counts, nbytes=nbytes)
        return out, counts, nbytes
    if op == "decode":
        mode = aw.DECODE_DENSE if st["case"]["mode"] == "dense" else aw.DECODE_INPLACE
        outs = aw.awsrc_decode_apply(prm, st["mods"], st["records"][0], -1, outs=st["out"], mode=mode, workspace=st["ws"])
        st["ws"] = outs[0]._awsrc_workspace
        return outs
    if op == "rtn":
        st["out"] = aw.awsrc_rtn_quantize_batch(st["Ws"], sdq=st["case"]["sdq"], outs=st["out"])
        return st["out"]
    return aw.awsrc_packed_gemv_batch(prm, st["shapes"], st["tasks"], sidecar=st["sidecar"])


# ------------------------------------------------------------------ exact --

def _mix(x, n):
    """Output n of the SplitMix64 stream at state x (arrays of uint64)."""
    with np.errstate(over="ignore"):
        z = x + np.uint64(n) * np.uint64(0x9E3779B97F4A7C15)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        return z ^ (z >> np.uint64(31))


def _signs(C, P, S):
    """The +-1 entries of every selector's basis (generator seed 0): S x C x P."""
    rows = np.arange(S)
    with np.errstate(over="ignore"):
        state = (rows.astype(np.uint64) + np.uint64(1)) * np.uint64(0x9E3779B97F4A7C15)
    key = _mix(state, 0)
    words = -(-C // 64)
    sign = [_mix(key, n + 1) for n in range(words)]
    n = words
    perm = np.tile(np.arange(C), (S, 1))
    for i in range(C - 1, 0, -1):
        n += 1
        k = (((_mix(key, n) >> np.uint64(32)) * np.uint64(i + 1)) >> np.uint64(32)).astype(np.int64)
        t = perm[rows, k].copy()
        perm[rows, k] = perm[:, i]
        perm[:, i] = t
    pool = np.tile(np.arange(C), (S, 1))
    out = np.empty((S, C, P))
    sg = np.stack([(sign[j // 64] >> np.uint64(j % 64)) & np.uint64(1) for j in range(C)], 1).astype(np.int64)
    for p in range(P):
        n += 1
        k = p + (((_mix(key, n) >> np.uint64(32)) * np.uint64(C - p)) >> np.uint64(32)).astype(np.int64)
        t = pool[rows, k].copy()
        pool[rows, k] = pool[:, p]
        pool[:, p] = t
        x = perm & pool[:, p][:, None]
        for s in (4, 2, 1):
            x = x ^ (x >> s)
        out[:, :, p] = 1 - 2 * ((sg + x) & 1)
    return torch.from_numpy(out).to(DEV)


def _residual(case, records):
    """(tile, residual of its C elements) of every record, in 64 bits."""
    _, tile, seed, scale, code = records
    sg = _signs(case["C"], case["P"], case["S"])
    if case["scale"] == "pow2":
        sc = torch.exp2(scale.double())
    else:
        sc = scale.to(torch.int16).view(torch.float16).double()
    r = torch.empty(tile.numel(), case["C"], dtype=torch.float64, device=DEV)
    for k in range(0, tile.numel(), 1 << 18):
        e = slice(k, k + (1 << 18))
        r[e] = torch.einsum("kcp,kp->kc", sg[seed[e]], code[e].double()) * (sc[e] / math.sqrt(case["C"]))[:, None]
    return tile, r


def _add_residual(case, records, mats):
    """The records' residuals added to 64-bit matrices, in place."""
    tile, r = _residual(case, records)
    off = 0
    for m in mats:
        v = m.view(-1, case["C"])
        at = (tile >= off) & (tile < off + v.shape[0])
        v.index_add_(0, tile[at] - off, r[at])
        off += v.shape[0]
    return mats


def exact(case, seed):
    """Outputs in 64 bits; the encoder's candidates and the stream are bytes and have none."""
    if case["op"] in ("encode", "select"):
        return None
    st = prepare(case, seed)
    if case["op"] == "decode":
        return _add_residual(case, st["records"], [m["W0"].double() for m in st["mods"]])
    if case["op"] == "rtn":
        out = []
        for W in st["Ws"]:
            r = _rtn(W, case["sdq"], torch.float64)
            out.append({k: (r[k] if k in ("W0", "sdq_consts") else None) for k in r})
        return out
    mats = []
    for (rows, cols), p in zip(st["shapes"], st["packed"]):
        c = p["codes"].to(torch.int64)
        q = torch.stack([c & 15, c >> 4], 1).reshape(-1)
        q = (q - 16 * (q > 7)).double().reshape(-1, 128)
        if case["sdq"]:
            k = p["sdq_consts"].double().reshape(-1, 2)[torch.arange(q.shape[0], device=DEV) // 256]
            s = k[:, 0] + p["sdq_codes"].double() * k[:, 1]
        else:
            s = p["scales"].view(torch.float16).double()
        mats.append((q * s[:, None]).reshape(rows, cols))
    _add_residual(case, st["records"], mats)
    return [t[2].double() @ m.T for t, m in zip(st["tasks"], mats)]
