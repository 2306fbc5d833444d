"""The work that a program using libkvq has it do, as a list of cases that can be prepared, run and compared.

A case names one pass through the public entry points (``op``) and its sizes:

  append     kvq_append      one new row per stream into the caches, position given by the host
  append_at  kvq_append_at   the same, position in device memory
  flush      kvq_flush_block ``rows`` new rows per stream into the int4 caches and the dequantized-prefix cache
  encode     kvq_encode      the bulk write after a prefill
  decode     kvq_decode      the full-prefix read of a decode step
  step       kvq_append + kvq_decode of the whole cache: one decode step
  roundtrip  kvq_encode + kvq_decode: quantize-dequantize, as accuracy experiments use the library
  calibrate  kvq_calibrate_lambda: one pass over calibration vectors

``streams * rows`` vectors of head dimension ``D`` go through a pass (``rows`` = 1 for the appends; of a step, ``rows`` is
the length of the cache that is read).  ``n_lambda`` lambda rows share the streams, ``streams / n_lambda`` (rounded up)
each: one per (layer, K or V) in a model.
"""
from __future__ import annotations

import math

import torch

from paper_2605_05699_b200 import binding as kb
from paper_2605_05699_b200 import workloads as wl

MODES = {"f16": torch.float16, "bf16": torch.bfloat16}
LARGEST_BYTES = 688_000_000   # one pass of the largest listed case


def _case(name, op, D, dtype, streams, rows, n_lambda, kind="gaussian", cache_rows=0, group=32, bits=4, rotated=False):
    c = {"op": op, "D": D, "dtype": dtype, "streams": streams, "rows": rows, "n_lambda": n_lambda, "kind": kind,
         "cache_rows": cache_rows or rows, "group": group, "bits": bits, "rotated": rotated}
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the write of one decode step in one layer of a 70B-sized model, batch 4: 32 K and 32 V streams
        _case("append_layer", "append", 128, "f16", 64, 1, 2, cache_rows=4096),
        # the same write for all 80 layers in one call, a lambda row per (layer, K / V)
        _case("append_model", "append", 128, "f16", 5120, 1, 160, cache_rows=256),
        # a full window of 16 tokens per stream leaves the fp16 window of one layer
        _case("flush_window", "flush", 128, "f16", 64, 16, 2, cache_rows=2048),
        # one decode step of a 1.5B-sized model that re-reads its whole prefix: 28 layers x 2 KV heads x (K, V)
        _case("step_1p5b", "step", 128, "f16", 112, 1152, 56, kind="k_outlier"),
        # prefill of one layer of the 70B-sized model at 32,768 tokens, batch 4
        _case("prefill_70b_layer", "encode", 128, "f16", 64, 32768, 2, kind="k_outlier"),
        # full-prefix read of that layer in a decode step
        _case("prefix_70b_layer", "decode", 128, "f16", 64, 32768, 2),
        # prefill of a 1B-sized model with head dimension 256 at 4096 tokens: all 26 layers in one call
        _case("prefill_1b", "encode", 256, "bf16", 52, 4096, 52, kind="k_outlier"),
        # full-prefix read of that model's cache
        _case("prefix_1b", "decode", 256, "bf16", 52, 4096, 52),
        # quantize-dequantize at a mixed-radix head dimension, as perplexity runs do on the fly
        _case("roundtrip_d96", "roundtrip", 96, "f16", 1, 65536, 1, kind="lognormal"),
        # the other mixed-radix head dimension, bf16, a ragged number of rows
        _case("roundtrip_d160", "roundtrip", 160, "bf16", 3, 33331, 3, kind="lognormal"),
        # a long prompt goes into the int4 cache and the dequantized-prefix cache block by block
        _case("flush_prefill", "flush", 128, "bf16", 64, 2000, 2, kind="k_outlier", cache_rows=4096),
        # the base quantizer (byte codes, one scale per vector): full-prefix read
        _case("prefix_bytes", "decode", 128, "bf16", 37, 8191, 1, group=128, bits=8),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["append", "append_at", "flush", "flush", "encode", "encode", "encode", "decode", "decode", "decode", "step",
                     "roundtrip", "calibrate"])
    D = rng.choice([64, 96, 128, 128, 160, 256, 256])
    dtype = rng.choice(["f16", "bf16"])
    if op == "calibrate" and D == 160:
        dtype = "f16"   # the only type this entry point takes at D = 160
    group, bits = rng.choice([(32, 4)] * 7 + [(D, 4), (32, 8), (D, 8)])
    kind = rng.choice(["gaussian", "lognormal", "k_outlier"])
    rotated = bits == 4 and op in ("append", "encode", "decode", "roundtrip") and rng.random() < 0.15
    passes = 2 if op in ("step", "flush", "roundtrip") else 1
    room = LARGEST_BYTES * (0.5 if D > 128 else 0.8) / passes
    if bits == 8 and dtype == "bf16" and D > 128:
        room /= 8       # served by the register FFT
    most = int(room / _vector_bytes(D, group, bits))
    if op in ("append", "append_at"):
        streams, rows, cache_rows = _log_uniform(rng, 1, 8192), 1, _log_uniform(rng, 64, 512)
        n_lambda = rng.choice([1, 2, max(1, streams // 32)])
    elif op == "flush":
        streams = _log_uniform(rng, 2, 128)
        rows = _log_uniform(rng, 8, min(4096, most // streams))
        cache_rows = rows + _log_uniform(rng, 1, 1024)
        n_lambda = rng.choice([1, 2, streams])
    elif op == "calibrate":
        streams, rows, n_lambda = 1, _log_uniform(rng, 2000, min(most, 500_000)), 1
        cache_rows = rows
    else:
        n = _log_uniform(rng, 500 if op != "step" else 4000, most)
        streams = min(_log_uniform(rng, 1, 128), n // 64 + 1)
        rows = n // streams
        cache_rows = rows
        n_lambda = rng.choice([1, 2, streams])
    return _case("", op, D, dtype, streams, rows, min(n_lambda, streams), kind, cache_rows, group, bits, rotated)


def _vector_bytes(D, group, bits):
    """Bytes of one vector in half precision and stored."""
    return 2 * D + _stored_bytes(D, group, bits)


def _stored_bytes(D, group, bits):
    return D * bits // 8 + 2 * (D // group)


def _stored(n, c, seed, device):
    """n stored vectors as a cache holds them: codes and scales of coefficients that spread over the channels like those of
    the transform (near-Gaussian, a persistent scale per channel), quantized against their group's largest."""
    D, g, q = c["D"], c["group"], 7 if c["bits"] == 4 else 127
    gen = torch.Generator(device=device)
    gen.manual_seed(seed)
    packed = torch.empty(n, D * c["bits"] // 8, dtype=torch.uint8, device=device)
    scales = torch.empty(n, D // g, dtype=torch.float16, device=device)
    width = torch.exp(0.5 * torch.randn(D, generator=gen, device=device))
    for at in range(0, n, 1 << 19):
        m = min(1 << 19, n - at)
        z = (torch.randn(m, D, generator=gen, device=device) * width).view(m, D // g, g)
        s = (z.abs().amax(-1) / q).to(torch.float16)
        codes = torch.round(z / s.float().unsqueeze(-1)).clamp_(-q, q).to(torch.int32).view(m, D)
        scales[at:at + m] = s
        if c["bits"] == 4:
            packed[at:at + m] = ((codes[:, 0::2] & 15) | ((codes[:, 1::2] & 15) << 4)).to(torch.uint8)
        else:
            packed[at:at + m] = (codes & 255).to(torch.uint8)
    return packed, scales


def prepare(case, seed):
    c, dev = case, torch.device("cuda", torch.cuda.current_device())
    D, S, R, T, dt = c["D"], c["streams"], c["rows"], c["cache_rows"], MODES[c["dtype"]]
    seed = 16 * seed + 1
    plan = kb.Plan(D, c["group"], 7, bits=c["bits"])
    if c["rotated"]:
        plan.set_rotation(wl.make_rotation(D, 11))
    kb.kvq_plan_prepare(plan.handle, dt, dev)
    spl = -(-S // c["n_lambda"])
    st = {"op": c["op"], "plan": plan, "h": plan.handle, "spl": spl, "rpl": spl * R,
          "lam": wl.make_lambda(c["n_lambda"], D, seed + 1, device=dev)}

    def vectors(n):
        return wl.make_vectors(n, D, c["dtype"], c["kind"], seed + 2, device=dev)

    op = c["op"]
    if op in ("append", "append_at", "flush"):
        st["pos"] = T - R
        st["pos_device"] = torch.tensor([T - R], dtype=torch.int64, device=dev)
        st["x"] = vectors(S * R).view((S, D) if op != "flush" else (S, R, D))
        st["packed"] = torch.zeros(S, T, D * c["bits"] // 8, dtype=torch.uint8, device=dev)
        st["scales"] = torch.zeros(S, T, D // c["group"], dtype=torch.float16, device=dev)
        # the caches, and beside them the rows that the call writes
        st["outputs"] = [st["packed"], st["scales"], st["packed"][:, T - R:], st["scales"][:, T - R:]]
        if op == "flush":
            st["dq"] = torch.zeros(S, T, D, dtype=dt, device=dev)
            st["outputs"] += [st["dq"], st["dq"][:, T - R:]]
    elif op == "step":
        packed, scales = _stored(S * R, c, seed + 3, dev)
        st["x"] = vectors(S)
        st["pos"] = R - 1
        st["packed"], st["scales"] = packed.view(S, R, -1), scales.view(S, R, -1)
        st["out"] = torch.empty(S, R, D, dtype=dt, device=dev)
        st["outputs"] = [st["packed"][:, R - 1], st["scales"][:, R - 1], st["out"]]
    elif op == "decode":
        st["packed"], st["scales"] = _stored(S * R, c, seed + 3, dev)
        st["out"] = torch.empty(S * R, D, dtype=dt, device=dev)
        st["outputs"] = [st["out"]]
    elif op == "calibrate":
        st["x"] = vectors(R)
        st["lambda_out"] = torch.empty(D, dtype=torch.float32, device=dev)
        st["outputs"] = [st["lambda_out"]]
    else:   # encode, roundtrip
        st["x"] = vectors(S * R)
        st["packed"], st["scales"] = plan.empty_packed(S * R, dev), plan.empty_scales(S * R, dev)
        st["outputs"] = [st["packed"], st["scales"]]
        if op == "roundtrip":
            st["out"] = torch.empty_like(st["x"])
            st["outputs"].append(st["out"])
    return st


def run(st):
    op, h, lam = st["op"], st["h"], st["lam"]
    if op == "append":
        kb.kvq_append(h, st["x"], lam, st["packed"], st["scales"], st["pos"], st["spl"])
    elif op == "append_at":
        kb.kvq_append_at(h, st["x"], lam, st["packed"], st["scales"], st["pos_device"], st["spl"])
    elif op == "flush":
        kb.kvq_flush_block(h, st["x"], lam, st["packed"], st["scales"], st["dq"], st["pos"], st["spl"])
    elif op == "encode":
        kb.kvq_encode(h, st["x"], lam, st["packed"], st["scales"], st["rpl"])
    elif op == "decode":
        kb.kvq_decode(h, st["packed"], st["scales"], lam, st["out"], st["rpl"])
    elif op == "step":
        kb.kvq_append(h, st["x"], lam, st["packed"], st["scales"], st["pos"], st["spl"])
        kb.kvq_decode(h, st["packed"], st["scales"], lam, st["out"], st["rpl"])
    elif op == "roundtrip":
        kb.kvq_encode(h, st["x"], lam, st["packed"], st["scales"], st["rpl"])
        kb.kvq_decode(h, st["packed"], st["scales"], lam, st["out"], st["rpl"])
    else:
        kb.kvq_calibrate_lambda(h, st["x"], st["lambda_out"])
    return st["outputs"]


def work(case):
    """Each half-precision row read or written once, each stored row written or read once, each lambda row once; the
    arithmetic of a real FFT of length D and of the quantizer, per direction."""
    c = case
    D, S, R = c["D"], c["streams"], c["rows"]
    half, stored = 2 * D, _stored_bytes(D, c["group"], c["bits"])
    per_vector = 2.5 * D * math.log2(D) + 8 * D
    n, op = S * R, c["op"]
    if op == "flush":
        moved, turns = n * (2 * half + stored), 2 * n           # what is dequantized is at hand: the codes are not read back
    elif op == "step":
        moved, turns = (S + n) * (half + stored), S + n
    elif op == "roundtrip":
        moved, turns = n * (2 * half + stored), 2 * n
    elif op == "calibrate":
        moved, turns = n * half, n
    else:
        moved, turns = n * (half + stored), n
    return {"bytes": moved + 4 * D * c["n_lambda"], "flops": turns * per_vector}


def tolerance(case):
    """About four times what the library differs by from the same arithmetic in 64 bits (listed cases and thirty drawn ones).

    Stored scales: one fp16 ulp on up to 3e-4 (fp16 input) or 2e-3 (bf16) of them, 4e-5 in the 2-norm.  Stored bytes: codes at
    rounding ties, up to 1.6e-5 of the bytes with 4-bit codes and 2.4e-5 with 8-bit ones.  Decoded rows: 3.9e-4 in fp16 (its
    operands are rounded to fp16 once), 6.4e-5 in bf16 (roundings that flip, each one ulp of 7.8e-3).  Where a pass decodes
    what it encoded, a code at a tie moves its row by about 0.03 of the row's norm, on up to 2e-3 of the rows."""
    op, f16 = case["op"], case["dtype"] == "f16"
    if op == "calibrate":
        return {"rel": 1e-5}
    differ = 6e-5 if case["bits"] == 4 else 1e-4
    # a call of a few rows: two of its bytes
    written = case["streams"] * (1 if op == "step" else case["rows"]) * case["D"] * case["bits"] // 8
    differ = min(0.01, max(differ, 2.0 / written))
    if op in ("flush", "roundtrip"):
        return {"rel": 2e-3 if f16 else 5e-3, "max": 0.1, "differ": differ}
    if op in ("decode", "step"):
        return {"rel": 1.6e-3 if f16 else 2.5e-4, "max": 1.6e-2, "differ": 0.0 if op == "decode" else differ}
    return {"rel": 1.6e-4, "max": 4e-3, "differ": differ}
