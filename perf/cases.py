"""The work that a user of the residual-VQ library has it do, as cases that can be timed and compared.

A case is one call of a public entry point on the data that it meets in use:

  encode     new keys or values go into the compressed cache (one token of a decode step ... a long prompt)
  decode     cached vectors come back as 16- or 32-bit vectors (one page ... a whole long cache)
  rope       cached keys come back rotated to their positions
  attention  one new token attends over the compressed cache
  learn      one step of codebook learning on a batch

Shapes are those of the repository's workloads (head dimension 128 or 256, groups of 32 channels, 8 key/value
heads, depth 4 ... 8, 256 ... 2048 codes per stage, codes as uint16 or packed).  Keys have heavy-tailed channel
scales with a few outlier channels, and strided groups; values are Gaussian, with contiguous groups; codebooks
shrink from stage to stage as learnt residual codebooks do.
"""
import math

import torch

import paper_2410_15704_b200 as rvq

HEADS = 8
GROUP = 32
OUTLIERS = 8                      # outlier channels of a key head
DECAY, EPS = 0.99, 1e-5
ROPE_BASE = 500000.0
DTYPES = {"bf16": rvq.BF16, "f16": rvq.F16, "f32": rvq.F32}


def _case(op, tokens, data, codes, depth=8, packed=False, dtype="bf16", dim=128, **more):
    return dict(op=op, tokens=tokens, data=data, codes=codes, depth=depth, packed=packed, dtype=dtype, dim=dim, **more)


def listed():
    cases = {
        # one sequence in its decode step: the new token's keys of one layer
        "encode_one_token": _case("encode", 1, "keys", 2048, packed=True),
        # a decode step of 77 sequences: the new tokens' values of one layer
        "encode_step_of_77": _case("encode", 77, "values", 2048, packed=True, dtype="f16"),
        # a prompt of 4096 tokens: its keys
        "encode_prompt_keys": _case("encode", 4096, "keys", 1024),
        # a small float32 batch on small codebooks
        "encode_float32": _case("encode", 512, "values", 256, dtype="f32"),
        # a long context's values at the default codebook size, packed as they are stored
        "encode_long_values": _case("encode", 32768, "values", 2048, packed=True),
        # a page of the cache read back
        "decode_page": _case("decode", 64, "values", 2048, packed=True),
        # that long context's values read back
        "decode_long_values": _case("decode", 32768, "values", 2048, packed=True),
        # a 128K-token cache read back, codes as uint16
        "decode_whole_cache": _case("decode", 131072, "values", 1024),
        # keys of a ragged context read back and rotated (half-split pairs)
        "rope_keys": _case("rope", 30001, "keys", 1024, pairing="halves"),
        # one new token over a short cache, and over a 128K-token one
        "attention_short": _case("attention", 1000, "keys", 1024, q_heads=32, pairing="halves"),
        "attention_long": _case("attention", 131072, "keys", 1024, q_heads=32, pairing="halves"),
        # one learning step on the largest batch that the repository trains on
        "learn_batch": _case("learn", 131072, "keys", 1024),
    }
    return [dict(c, name=name) for name, c in cases.items()]


#: (row, stage, code) triples of the largest listed encode: the bound of the drawn ones
_MOST_SCORES = 131072 * HEADS * 4 * 8 * 1024
#: bytes of the largest listed decode's output
_MOST_OUT = 131072 * HEADS * 128 * 2


def _log_int(rng, low, high):
    return min(high, max(low, int(round(math.exp(rng.uniform(math.log(low), math.log(high)))))))


def draw(rng):
    op = rng.choice(["encode", "encode", "decode", "decode", "rope", "attention", "learn"])
    data = "keys" if op in ("rope", "attention") else rng.choice(["keys", "values"])
    dim = 128 if op == "attention" else rng.choice([128, 128, 128, 256])
    depth = rng.choice([4, 6, 8, 8, 8])
    dtype = rng.choice(["bf16", "bf16", "f16", "f32"])
    packed = rng.random() < 0.5
    codes = rng.choice([256, 512, 1000, 1024, 1024] + ([2048, 2048] if op != "attention" else []))
    rows = HEADS * (dim // GROUP)                              # group rows of a token
    more = {}
    if op in ("encode", "learn"):
        most = min(131072, _MOST_SCORES // (rows * depth * codes))
        tokens = _log_int(rng, 1 if op == "encode" else 256, most)
    elif op in ("decode", "rope"):
        tokens = _log_int(rng, 1, min(131072, _MOST_OUT // (HEADS * dim * (4 if dtype == "f32" else 2))))
    else:
        tokens = _log_int(rng, 64, 131072)
        more["q_heads"] = rng.choice([8, 16, 32])
    if op in ("rope", "attention"):
        more["pairing"] = rng.choice(["halves", "adjacent"])
    return _case(op, tokens, data, codes, depth=depth, packed=packed, dtype=dtype, dim=dim, **more)


# ------------------------------------------------------------------------------------------------ shapes

def _vectors(case):
    return case["tokens"] * HEADS


def _groups(case):
    return case["dim"] // GROUP


def _config(case, data=None):
    layout = rvq.STRIDED if (data or case["data"]) == "keys" else rvq.CONTIGUOUS
    bits = max(1, (case["codes"] - 1).bit_length()) if case["packed"] else 16
    return rvq.make_config(case["dim"], GROUP, layout, case["depth"], case["codes"], bits, DTYPES[case["dtype"]], 0)


def _code_bytes(case):
    bits = (case["codes"] - 1).bit_length() if case["packed"] else 16
    return (_groups(case) * case["depth"] * bits + 31) // 32 * 4


def work(case):
    """Each input read once and each output written once; two operations for every multiply-add."""
    n, G, R, K, dim = _vectors(case), _groups(case), case["depth"], case["codes"], case["dim"]
    elem = 4 if case["dtype"] == "f32" else 2
    books = R * K * GROUP * 4
    x, cache = n * dim * elem, n * (_code_bytes(case) + 2)
    scores = 2.0 * GROUP * K * R * G * n
    op = case["op"]
    if op == "encode":
        return {"bytes": x + cache + books, "flops": scores}
    if op == "decode":
        return {"bytes": cache + x + books, "flops": float(n * dim * (R + 1))}
    if op == "rope":
        return {"bytes": cache + x + books + case["tokens"] * (dim // 2 * 8 + 4), "flops": float(n * dim * (R + 4))}
    if op == "attention":
        per_value = 2 * (R + 1) + 3 + 4 * case["q_heads"] // HEADS      # both sums, the rotation, both products
        return {"bytes": 2 * (cache + books) + case["tokens"] * (dim // 2 * 8) + 2 * case["q_heads"] * dim * 4,
                "flops": float(n * dim * per_value)}
    state = R * K * (GROUP + 1) * 4
    return {"bytes": x + cache + 2 * (books + state), "flops": scores + float(n * dim * R)}


def tolerance(case):
    op = case["op"]
    if op == "encode":
        return "exact"                    # the nearest code under float32 arithmetic; binary16 deviations
    if op in ("decode", "rope"):
        return {"rel": {"bf16": 4e-3, "f16": 1e-3, "f32": 1e-5}[case["dtype"]]}
    if op == "attention":
        return {"rel": 5e-5}              # float32 sums over the tokens, and exponentials of float32 scores
    # float32 sums of the rows of a code; a row at equal distance from two codes may go to either, which
    # moves both and, from then on, everything that follows from them
    return {"rel": 1e-4, "max": 0.2, "differ": 1e-3}


# ------------------------------------------------------------------------------------------------ inputs

def _channel_scales(gen, data, dim):
    """[heads][dim] scales of the channels: 1 for values; heavy-tailed with a few outliers for keys."""
    if data == "values":
        return torch.ones(HEADS, dim, device="cuda")
    u = torch.rand(HEADS, dim, generator=gen, device="cuda").clamp_min(1e-7)
    a = 0.25 - torch.log(u)                                   # 0.25 + |Laplace(0, 1)|
    outlier = torch.rand(HEADS, dim, generator=gen, device="cuda").argsort(dim=1)[:, :OUTLIERS]
    return a.scatter(1, outlier, a.gather(1, outlier) * 20.0)


def _inputs(gen, case, data):
    """The head vectors [tokens * heads][dim] of a batch and codebooks [depth][codes][32] that fit them."""
    dim, G, R, K = case["dim"], _groups(case), case["depth"], case["codes"]
    a = _channel_scales(gen, data, dim)
    x = torch.randn(case["tokens"], HEADS, dim, generator=gen, device="cuda").mul_(a).view(-1, dim)
    x = x.to(rvq.TORCH_DTYPE[DTYPES[case["dtype"]]])
    # codewords of stage r: group vectors of this distribution in scaled units, 0.8^r as large
    unit = a / a.square().mean(dim=1, keepdim=True).sqrt()
    groups = (unit.view(HEADS, GROUP, G).transpose(1, 2) if data == "keys" else unit.view(HEADS, G, GROUP)).reshape(-1, GROUP)
    pick = torch.randint(groups.shape[0], (R, K), generator=gen, device="cuda")
    books = torch.randn(R, K, GROUP, generator=gen, device="cuda") * groups[pick]
    books *= (0.8 ** torch.arange(R, device="cuda", dtype=torch.float32)).view(R, 1, 1)
    return x, books.contiguous()


def _encode(cfg, x, n, b):
    rvq.rvq_encode(cfg, x, n, cfg.dim, b.codebooks, b.prepared, b.codes, b.std, b.workspace, b.workspace_bytes, b.status)


def _cache(gen, case, data):
    """A compressed cache: the buffers of a quantizer whose codes and deviations are those of a drawn batch."""
    cfg, n = _config(case, data), _vectors(case)
    x, books = _inputs(gen, case, data)
    b = rvq.alloc_buffers(cfg, n, books)
    _encode(cfg, x, n, b)
    return cfg, b


def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    n, R, K, dim, op = _vectors(case), case["depth"], case["codes"], case["dim"], case["op"]
    s = {"op": op, "n": n, "case": case}
    if op in ("encode", "learn"):
        s["cfg"] = _config(case)
        s["x"], books = _inputs(gen, case, case["data"])
        s["b"] = rvq.alloc_buffers(s["cfg"], n, books)
        if op == "learn":
            s["count"] = torch.full((R, K), n * _groups(case) / K, device="cuda")      # a state under way: N rows a code
            s["sum"] = s["b"].codebooks * s["count"].unsqueeze(2)
            s["energy"] = torch.empty(R, device="cuda")
    elif op in ("decode", "rope"):
        s["cfg"], s["b"] = _cache(gen, case, case["data"])
        s["out"] = torch.empty(n, dim, dtype=rvq.TORCH_DTYPE[s["cfg"].x_dtype], device="cuda")
    else:
        s["cfg"], s["b"] = _cache(gen, case, "keys")
        s["cfg_v"], s["v"] = _cache(gen, case, "values")
        s["q"] = torch.randn(case["q_heads"], dim, generator=gen, device="cuda")
        s["ws_bytes"] = rvq.rvq_attention_workspace_bytes(case["tokens"], case["q_heads"])
        s["ws"] = torch.empty(s["ws_bytes"], dtype=torch.uint8, device="cuda")
        s["out"] = torch.empty(case["q_heads"], dim, device="cuda")
    if op in ("rope", "attention"):
        s["pairing"] = rvq.ROPE_HALVES if case["pairing"] == "halves" else rvq.ROPE_ADJACENT
        s["table"] = torch.empty(case["tokens"], dim // 2, 2, device="cuda")
        rvq.rvq_rope_table(dim, ROPE_BASE, case["tokens"], s["table"])
        s["position"] = torch.arange(case["tokens"], dtype=torch.int32, device="cuda")
    return s


# ------------------------------------------------------------------------------------------------ calls

def run(s):
    op, cfg, b, n, case = s["op"], s["cfg"], s["b"], s["n"], s["case"]
    if op == "encode":
        _encode(cfg, s["x"], n, b)
        return {"codes": b.codes, "std": b.std}
    if op == "decode":
        rvq.rvq_decode(cfg, b.codes, b.std, n, b.codebooks, b.prepared, s["out"], cfg.dim, b.status)
        return s["out"]
    if op == "rope":
        rvq.rvq_decode_rope(cfg, b.codes, b.std, n, b.codebooks, b.prepared, s["position"], HEADS, s["table"],
                            case["tokens"], s["pairing"], s["out"], cfg.dim, b.status)
        return s["out"]
    if op == "attention":
        v = s["v"]
        rvq.rvq_attention_decode(cfg, s["cfg_v"], s["q"], case["q_heads"], b.codes, b.std, v.codes, v.std, case["tokens"],
                                 HEADS, b.codebooks, v.codebooks, s["position"], s["table"], case["tokens"], s["pairing"],
                                 cfg.dim ** -0.5, s["out"], s["ws"], s["ws_bytes"], b.status)
        return s["out"]
    rvq.rvq_learn_step(cfg, s["x"], n, cfg.dim, b.codebooks, b.prepared, s["count"], s["sum"], b.codes, b.std, DECAY, EPS,
                       b.workspace, b.workspace_bytes, b.status, stage_energy=s["energy"])
    return {"codes": b.codes, "std": b.std, "codebooks": b.codebooks, "count": s["count"], "sum": s["sum"],
            "energy": s["energy"]}
