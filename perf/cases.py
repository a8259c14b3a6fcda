"""Performance cases: what a program that keeps its KV cache in this codec asks of it.

A case is a call (or an encode and the decode that follows it) on one cache shape, through the
package's public functions, with buffers the program allocated once. Inputs are seeded
synthetic caches drawn on the GPU with the value structure of ``synth.py``: keys with
per-channel scales and a few outlier channels, values with per-token scales, gauges
exp(A - A^T). Packed inputs of the reading calls (decode, attention) are drawn as bell-shaped
codes with a scale and a zero per block, so they do not depend on the encoder.
"""
import math

import torch

import paper_2607_20538_gb300 as cg

BACKEND = {"rows": cg.CG_BLOCK_UNIFORM, "kivi": cg.CG_KIVI, "tiles": cg.CG_BLOCK_TILE}
DEVICE = "cuda"


def _case(name, op, L, B, H, T, d=128, group=128, backend="rows", bits=4, block=64, residual=0, t0=0, T_cap=0, n_rep=0):
    return dict(name=name, op=op, L=L, B=B, H=H, T=T, d=d, group=group, backend=backend, bits=bits, block=block,
                residual=residual, t0=t0, T_cap=T_cap, n_rep=n_rep)


def listed():
    return [
        # the smallest use: one short prompt of a small model, compressed and read back
        _case("short_roundtrip", "roundtrip", 1, 1, 2, 256, d=64, group=16, block=32),
        # one token of 64 running sequences is added to every layer's 4-bit history
        _case("append_token", "encode", 32, 64, 8, 1, t0=1000, T_cap=1024),
        # a KIVI decode loop at 32k tokens: the appended token completes a key group
        _case("kivi_append", "kivi_append", 28, 4, 4, 1, group=64, backend="kivi", bits=3, block=128, residual=128,
              t0=32767, T_cap=32768),
        # one layer's decoding attention over 64 histories of 16k tokens, four query heads a KV head
        _case("batch_attention", "attention", 1, 64, 8, 16384, n_rep=4),
        # one layer's decoding attention of a single long 8-bit sequence of odd length
        _case("long_attention", "attention", 1, 1, 8, 32767, bits=8, n_rep=4),
        # a prefilled cache of 32 layers and 8k tokens, compressed at 4 bits
        _case("prefill_encode", "encode", 32, 1, 8, 8192),
        # and restored
        _case("prefill_decode", "decode", 32, 1, 8, 8192),
        # the largest cache: 46 layers, 16 KV heads, two sequences, 6 bits, small groups and blocks
        _case("large_encode", "encode", 46, 2, 16, 8192, group=32, bits=6, block=32),
        # KIVI at 3 bits over 32k tokens: a prefill compressed
        _case("kivi_encode", "encode", 28, 4, 4, 32768, group=64, backend="kivi", bits=3, block=128, residual=128),
        # and restored
        _case("kivi_decode", "decode", 28, 4, 4, 32768, group=64, backend="kivi", bits=3, block=128, residual=128),
        # the paper's block shape, one range per 16 tokens x 128 channels, on a prefilled cache
        _case("tile_encode", "encode", 32, 1, 8, 8192, backend="tiles", block=128),
        # the Hadamard control without a gauge tensor: compressed and read back
        _case("hadamard_roundtrip", "hadamard", 32, 1, 8, 8192),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["encode", "encode", "decode", "decode", "tiles", "kivi", "kivi", "append", "kivi_append",
                     "attention", "attention", "hadamard", "roundtrip"])
    bits = rng.choice([2, 3, 4, 4, 6, 8])
    H = rng.choice([1, 2, 4, 8, 16])
    group = rng.choice([16, 32, 64, 128, 128])
    block = rng.choice([32, 64, 64, 128])
    if op == "attention":
        B, T = _log(rng, 1, 64), _log(rng, 100, 32768)
        T = max(1, min(T, (1 << 24) // (B * H)))
        return _case("", "attention", 1, B, H, T, group=group, bits=bits, block=block, n_rep=rng.choice([1, 2, 4, 4, 8]),
                     backend=rng.choice(["rows", "rows", "tiles"]))
    if op == "kivi_append":
        L, B, H = rng.randint(1, 32), rng.randint(1, 8), rng.choice([2, 4, 8])
        R, cap = rng.choice([0, 32, 128]), _log(rng, 1024, 16384) // 128 * 128
        t0 = rng.randint(256, cap - 17)
        if rng.random() < 0.5:  # half of them complete a key group
            t0 = min(cap - 17, (t0 - R) // 128 * 128 + R + 127)
        return _case("", "kivi_append", L, B, H, rng.choice([1, 1, 2, 16]), group=rng.choice([32, 64, 128]), backend="kivi",
                     bits=rng.choice([2, 3, 4]), block=128, residual=R, t0=t0, T_cap=cap)
    if op == "append":
        L, B, cap = rng.randint(1, 32), _log(rng, 1, 64), _log(rng, 64, 1024)
        cap = max(64, min(cap, (1 << 24) // (L * 2 * B * H)))  # at most 2^24 token rows, or 64 a history
        return _case("", "encode", L, B, H, rng.choice([1, 1, 1, 4, 17]), group=group, bits=bits, block=block,
                     t0=rng.randint(0, cap - 17), T_cap=cap)
    # whole caches: at most 2^29 values, fewer for the head sizes other than 128
    d = 128 if op in ("tiles", "kivi") else rng.choice([64, 128, 128, 128, 256])
    most = 1 << 29 if d == 128 and op != "roundtrip" else 1 << 25
    T, B = _log(rng, 65, 32768), rng.randint(1, 4)
    H = max(1, min(H, most // (2 * B * T * d)))
    B = max(1, min(B, most // (2 * H * T * d)))
    L = max(1, min(rng.randint(1, 32), most // (2 * B * H * T * d)))
    group, block = min(group, d), min(block, d)
    if op == "tiles":
        return _case("", "encode", L, B, H, T, group=group, backend="tiles", bits=bits, block=block)
    if op == "kivi":
        return _case("", rng.choice(["encode", "decode"]), L, B, H, max(T, 300), group=rng.choice([32, 64, 128]), backend="kivi",
                     bits=rng.choice([2, 3, 4]), block=128, residual=rng.choice([0, 32, 128]))
    return _case("", op, L, B, H, T, d=d, group=group, bits=bits, block=block)


def _params(c):
    return cg.Params(BACKEND[c["backend"]], c["group"], c["bits"], c["block"], c["residual"])


def _shape(c):
    return cg.Shape(c["L"], c["B"], c["H"], c["T"], c["d"], c["t0"], c["T_cap"])


def _gen(seed):
    return torch.Generator(device=DEVICE).manual_seed(int(seed))


def _cache(c, T, gen):
    """bf16 [L][2][B][H][T][d], drawn layer by layer."""
    L, B, H, d = c["L"], c["B"], c["H"], c["d"]
    x = torch.empty((L, 2, B, H, T, d), dtype=torch.bfloat16, device=DEVICE)
    for l in range(L):
        ks = torch.empty((H, 1, d), device=DEVICE).log_normal_(0.0, 0.5, generator=gen)
        out = torch.rand((H, 1, d), device=DEVICE, generator=gen).topk(4, dim=-1).indices
        ks.scatter_(-1, out, ks.gather(-1, out) * 10.0)
        for b in range(B):
            x[l, 0, b] = torch.randn((H, T, d), device=DEVICE, generator=gen) * ks
            vs = torch.empty((H, T, 1), device=DEVICE).log_normal_(0.0, 0.3, generator=gen)
            x[l, 1, b] = torch.randn((H, T, d), device=DEVICE, generator=gen) * vs
    return x


def _gauges(c, gen):
    """fp32 [L][2][H][d/g][g][g]: exp(A - A^T)."""
    g = c["group"]
    a = torch.randn((c["L"] * 2 * c["H"] * (c["d"] // g), g, g), device=DEVICE, dtype=torch.float64, generator=gen)
    a *= 1.0 / math.sqrt(g)
    e = torch.matrix_exp(a - a.transpose(1, 2))
    return e.float().reshape(c["L"], 2, c["H"], c["d"] // g, g, g).contiguous()


def _draw_codes(n, bits, gen):
    """n codes (a multiple of 8) as bytes: bell-shaped, packed as a little-endian bit stream."""
    out = torch.empty((n // 8, bits), dtype=torch.uint8, device=DEVICE)
    qmax, step = (1 << bits) - 1, 1 << 23
    for i in range(0, n // 8, step):
        m = min(step, n // 8 - i)
        q = torch.randn((m, 8), device=DEVICE, generator=gen).mul_(qmax / 6).add_(qmax / 2).round_().clamp_(0, qmax).to(torch.int64)
        w = (q << (torch.arange(8, device=DEVICE) * bits)).sum(1)
        out[i:i + m] = ((w[:, None] >> (torch.arange(bits, device=DEVICE) * 8)) & 255).to(torch.uint8)
    return out.view(-1)


def _draw_scales(n, bits, gen):
    """n {scale, zero} pairs as int32 (two fp16 values each)."""
    qmax = (1 << bits) - 1
    s = torch.empty(n, device=DEVICE).log_normal_(0.0, 0.3, generator=gen).mul_(5.0 / qmax)
    m = s * (qmax / 2) * torch.randn(n, device=DEVICE, generator=gen).mul_(0.1).sub_(1.0)
    return torch.stack([s, m], 1).half().view(torch.int32).view(-1)


def _unpack(codes, bits):
    """Packed bytes (whole groups of 8 codes) -> codes as fp64."""
    b = codes.reshape(-1, bits).to(torch.int64)
    w = (b << (torch.arange(bits, device=DEVICE) * 8)).sum(1)
    return ((w[:, None] >> (torch.arange(8, device=DEVICE) * bits)) & ((1 << bits) - 1)).double().view(-1)


def _pair(scales):
    """int32 {scale, zero} pairs -> fp64 [..., 2]."""
    return scales.view(torch.float16).view(*scales.shape, 2).double()


def prepare(case, seed):
    c, gen = case, _gen(seed)
    shape, params, op = _shape(c), _params(c), c["op"]
    s = dict(op=op, shape=shape, params=params)
    units = c["L"] * 2 * c["B"] * c["H"]
    if op != "hadamard":
        s["gauges"] = _gauges(c, gen)
    if op == "attention":
        nc, ns, _ = cg.packed_bytes(shape, params)
        s["codes"], s["scales"] = _draw_codes(nc * 8 // c["bits"], c["bits"], gen), _draw_scales(ns // 4, c["bits"], gen)
        n = (c["L"], c["B"], c["H"], c["n_rep"], c["d"])
        # queries that give the logits a standard deviation of about 2.5, as trained attention has
        s["q"] = torch.randn(n, device=DEVICE, generator=gen).mul_(3.0).bfloat16()
        s["out"] = torch.empty(n, dtype=torch.float32, device=DEVICE)
        s["workspace"] = torch.empty(cg.attention_workspace_bytes(shape, params, c["n_rep"]), dtype=torch.uint8, device=DEVICE)
        s["n_rep"], s["scale"] = c["n_rep"], 1.0 / math.sqrt(c["d"])
        return s
    if op == "kivi_append":
        s["buffers"] = cg.kivi_stream_alloc(shape, params)
        ring = s["buffers"][2]
        ring.copy_(torch.randn(ring.numel(), device=DEVICE, generator=gen).bfloat16().view(torch.int16))
        s["kv"] = _cache(c, c["T"], gen)
        return s
    if op == "decode":
        nc, ns, nr = cg.packed_bytes(shape, params)
        s["codes"], s["scales"] = _draw_codes(nc * 8 // c["bits"], c["bits"], gen), _draw_scales(ns // 4, c["bits"], gen)
        s["residual"] = torch.randn(max(nr // 2, 8), device=DEVICE, generator=gen).bfloat16().view(torch.int16)
    else:
        s["kv"] = _cache(c, c["T"], gen)
        s["codes"], s["scales"], s["residual"] = cg.alloc_outputs(shape, params)
    if op != "encode":
        s["out"] = torch.empty((units, c["T"], c["d"]), dtype=torch.bfloat16, device=DEVICE)
    return s


def run(state):
    s = state
    op, shape, params = s["op"], s["shape"], s["params"]
    if op == "attention":
        cg.attention(shape, params, s["n_rep"], s["scale"], s["q"], s["codes"], s["scales"], s["gauges"], s["out"], s["workspace"])
        return {"out": s["out"]}
    if op == "kivi_append":
        codes, scales, ring, workspace = s["buffers"]
        cg.kivi_append(shape, params, s["kv"], s["gauges"], codes, scales, ring, workspace)
        return {"codes": codes, "scales": scales, "ring": ring}
    if op == "hadamard":
        cg.encode_hadamard(shape, params, s["kv"], s["codes"], s["scales"])
        cg.decode_hadamard(shape, params, s["codes"], s["scales"], s["out"])
        return {"codes": s["codes"], "scales": s["scales"], "out": s["out"]}
    got = {}
    if op in ("encode", "roundtrip"):
        cg.encode(shape, params, s["kv"], s["gauges"], s["codes"], s["scales"], s["residual"])
        got = {"codes": s["codes"], "scales": s["scales"]}
        if params.residual:
            got["residual"] = s["residual"]
    if op in ("decode", "roundtrip"):
        cg.decode(shape, params, s["codes"], s["scales"], s["residual"], s["gauges"], s["out"])
        got["out"] = s["out"]
    return got


def _n_quantized(c, T):
    R, G = c["residual"], c["block"]
    return T if c["backend"] != "kivi" else 0 if T <= R else (T - R) // G * G


def work(case):
    c = case
    L, B, H, T, d, g, bits = (c[k] for k in ("L", "B", "H", "T", "d", "group", "bits"))
    units, op = L * 2 * B * H, c["op"]
    gauges = 0 if op == "hadamard" else L * 2 * H * d * g * 4
    per_range = {"rows": 1, "tiles": 16, "kivi": 1}[c["backend"]]

    def packed(n):  # codes and scales of n tokens of every unit
        ranges = -(-n // per_range) * (d // c["block"])
        if c["backend"] == "kivi":
            ranges = n * d // c["block"]
        return units * (n * d * bits // 8 + ranges * 4)

    if op == "attention":
        rows = L * B * H * c["n_rep"]
        return {"bytes": packed(T) + gauges + rows * d * 6, "flops": rows * (T * d * 4 + 2 * d * g * 2)}
    if op == "kivi_append":
        done = _n_quantized(c, c["t0"] + T) - _n_quantized(c, c["t0"])
        moved = units * d * 2 * (2 * T + (done if done else 0))
        return {"bytes": moved + (packed(done) + gauges if done else 0), "flops": units * done * d * 2 * g}
    nq = _n_quantized(c, T)
    transform = 2 * g if op != "hadamard" else int(math.log2(g)) + 1
    one = units * (nq * d * 2 + (T - nq) * d * 4) + packed(nq) + gauges
    times = 2 if op in ("roundtrip", "hadamard") else 1
    return {"bytes": one * times, "flops": units * nq * d * transform * times}


def _hadamard(n):
    h = torch.ones((1, 1), dtype=torch.float64, device=DEVICE)
    while h.shape[0] < n:
        h = torch.cat([torch.cat([h, h], 1), torch.cat([h, -h], 1)], 0)
    return h / math.sqrt(n)


def _dequantized_rows(codes, scales, bits, n, d, block):
    """fp64 [n][d] of n token rows, one {scale, zero} per row and block."""
    sm = _pair(scales.reshape(n, d // block, 1))
    return (_unpack(codes, bits).view(n, d // block, block) * sm[..., 0] + sm[..., 1]).view(n, d)


def _rotated(z, G, back):
    """z [..., T, d] by the d/g gauges G [..., d/g, g, g] of its groups; back = G^T."""
    g = G.shape[-1]
    y = z.unflatten(-1, (-1, g)).transpose(-2, -3)  # [..., d/g, T, g]
    return (y @ (G if back else G.transpose(-1, -2))).transpose(-2, -3).flatten(-2)


def _exact_rows_roundtrip(x, G, bits, block):
    """Encode and decode of token rows [..., T, d] in fp64 (fp16 scale and zero)."""
    qmax = (1 << bits) - 1
    z = _rotated(x.double(), G, False).unflatten(-1, (-1, block))
    lo, hi = z.amin(-1, keepdim=True), z.amax(-1, keepdim=True)
    s, m = ((hi - lo) / qmax).half().double(), lo.half().double()
    q = torch.where(s > 0, ((z - m) / s).round().clamp(0, qmax), torch.zeros_like(z))
    return _rotated((q * s + m).flatten(-2), G, True)


def exact(case, seed):
    c, op = case, case["op"]
    if op in ("encode", "kivi_append"):
        return None  # codes, scales and raw tokens: whole numbers
    s = prepare(c, seed)
    L, B, H, T, d, bits, block = (c[k] for k in ("L", "B", "H", "T", "d", "bits", "block"))
    if op in ("roundtrip", "hadamard"):
        G = s["gauges"].double()[:, :, None] if op == "roundtrip" else _hadamard(c["group"]).expand(L, 2, 1, H, d // c["group"], -1, -1)
        out = torch.stack([_exact_rows_roundtrip(s["kv"][l], G[l], bits, block) for l in range(L)])
        return {"codes": None, "scales": None, "out": out.view(-1, T, d)}
    G = s["gauges"].double()
    if op == "attention":
        out = torch.empty((L, B, H, c["n_rep"], d), dtype=torch.float64, device=DEVICE)
        codes = s["codes"].view(L, 2, B, H, -1)
        scales = s["scales"].view(L, 2, B, H, -1, d // block)
        if c["backend"] == "tiles":
            scales = scales.repeat_interleave(16, dim=4)[..., :T, :]
        for l in range(L):
            for b in range(B):
                k, v = (_rotated(_dequantized_rows(codes[l, i, b].reshape(-1), scales[l, i, b].reshape(-1), bits, H * T, d, block)
                                 .view(H, T, d), G[l, i], True) for i in (0, 1))
                scale = float(torch.tensor(s["scale"], dtype=torch.float32))
                p = torch.softmax(scale * s["q"][l, b].double() @ k.transpose(1, 2), dim=-1)
                out[l, b] = p @ v
        return {"out": out}
    out = torch.empty((L, 2, B, H, T, d), dtype=torch.float64, device=DEVICE)
    nq = _n_quantized(c, T)
    if c["backend"] == "rows":
        codes, scales = s["codes"].view(L, 2, B * H * T, -1), s["scales"].view(L, 2, B * H * T, -1)
        for l in range(L):
            for i in (0, 1):
                z = _dequantized_rows(codes[l, i], scales[l, i], bits, B * H * T, d, block).view(B, H, T, d)
                out[l, i] = _rotated(z, G[l, i], True)
        return {"out": out.view(-1, T, d)}
    n, pay = B * H * nq, block * bits // 8  # KIVI: a layer's keys, then its values
    if nq:
        codes, scales = s["codes"].view(L, 2, -1), s["scales"].view(L, 2, -1)
        for l in range(L):
            ks = _pair(scales[l, 0].view(-1, d, 1))
            k = _unpack(codes[l, 0], bits).view(-1, d, block) * ks[..., 0] + ks[..., 1]
            k = k.view(B, H, nq // block, d, block).transpose(-1, -2).reshape(B, H, nq, d)
            out[l, 0, :, :, :nq] = _rotated(k, G[l, 0], True)
            v = _dequantized_rows(codes[l, 1], scales[l, 1], bits, n, d, block).view(B, H, nq, d)
            out[l, 1, :, :, :nq] = _rotated(v, G[l, 1], True)
    if T > nq:
        out[..., nq:, :] = s["residual"][: L * 2 * B * H * (T - nq) * d].view(torch.bfloat16).view(L, 2, B, H, T - nq, d).double()
    return {"out": out.view(-1, T, d)}
