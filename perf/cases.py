"""Timed workloads of the library: what its users call, over the sizes they call it with.

Every case goes through the public binding (`paper_1504_00353_gb300.polar`) with the launch
shapes that `autotune.shape_for` / `batch_shape` hand out, as `bench.py` and the examples do:
tuned shapes for the codes of the shape table, the library's own choice for any other code.
A case is a dict:

  path    "decode"  polar_decode / polar_decode_i8 on device LLRs
          "mixed"   polar_batch_decode: frames of the five mixed codes in one launch
          "sim"     one Monte-Carlo pass: random bits, encoder, AWGN channel, decoder, error count
          "host"    polar_decode_host: pinned host LLRs to pinned host bits
  N, K, design_db, ebn0_db   the code and its channel (not for "mixed")
  frames  frames of one pass;  dtype  "f32" or "i8" LLRs
  compiled  whether the program compiled the code's specialised decoder or runs the interpreter
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1504_00353_gb300 import autotune, polar, synth

DEV = "cuda"
MAX_ELEMS = 1 << 26  # frames * N of a drawn case


def _case(path, N, K, frames, dtype, design_db, ebn0_db, compiled=True, **kw):
    return dict(path=path, N=N, K=K, frames=frames, dtype=dtype, design_db=design_db,
                ebn0_db=ebn0_db, compiled=compiled, **kw)


def listed():
    return [
        # one short frame of a latency-bound link: launch and the serial chain are everything
        _case("decode", 2048, 1723, 1, "f32", 3.0, 3.0, name="one_n2048_f32"),
        # the paper's headline: the latency of one (32768, 29492) int8 frame
        _case("decode", 32768, 29492, 1, "i8", 4.0, 4.0, name="one_n32768_i8"),
        # a base-station batch of short rate-1/2 frames (the benchmark's first configuration)
        _case("decode", 1024, 512, 10000, "f32", 2.5, 2.5, name="batch_n1024_f32"),
        # a code the shape table does not hold, at the library's own shape; odd frame count
        _case("decode", 2048, 1707, 2001, "i8", 3.5, 3.5, name="batch_n2048_i8"),
        # the throughput configuration of the benchmark, both LLR types
        _case("decode", 32768, 29492, 4096, "i8", 4.0, 4.0, name="batch_n32768_i8"),
        _case("decode", 32768, 29492, 4096, "f32", 4.0, 4.0, name="batch_n32768_f32"),
        # the longest code of the benchmark (storage, quantum key distribution)
        _case("decode", 1 << 20, 880804, 64, "i8", 3.5, 3.5, name="batch_n1M_i8"),
        # traffic of five codes in one persistent launch, a quarter of the benchmark's batch
        dict(path="mixed", frames=16384, dtype="i8", ebn0_db=3.0, name="mixed_i8"),
        # a program that decodes at once, without compiling: the operation-list interpreter
        _case("decode", 1024, 512, 1000, "f32", 2.5, 2.5, compiled=False, name="interp_n1024_f32"),
        # error-rate simulation, short code in float32 and long code in int8
        _case("sim", 1024, 512, 16384, "f32", 2.5, 2.5, name="sim_n1024_f32"),
        _case("sim", 32768, 29492, 1024, "i8", 4.0, 4.5, name="sim_n32768_i8"),
        # the end-to-end call: frames in pinned host memory, bits back to host memory
        _case("host", 32768, 29492, 4096, "i8", 4.0, 4.0, name="host_n32768_i8"),
    ]


def draw(rng):
    path = rng.choice(["decode"] * 5 + ["mixed", "sim", "sim", "host"])
    dtype = rng.choice(["i8", "f32"])
    if path == "mixed":
        frames = int(round(2.0 ** rng.uniform(6, 14)))
        return dict(path=path, frames=frames, dtype=dtype, ebn0_db=round(rng.uniform(2.0, 4.5), 2))
    N = 1 << rng.randint(8, 15)
    K = int(round(N * rng.uniform(0.4, 0.92)))
    db = round(rng.uniform(2.0, 4.5), 2)
    compiled = path != "decode" or rng.random() < 0.8
    most = MAX_ELEMS // (1 if compiled else 8) // N // (2 if path == "sim" else 1)
    frames = int(round(2.0 ** rng.uniform(0 if path == "decode" else 5, math.log2(min(most, 20000)))))
    return _case(path, N, K, frames, dtype, db, db, compiled=compiled)


# ---------------------------------------------------------------- handles a program keeps

_codes: dict = {}
_batches: dict = {}


def _mask(N, K, design_db):
    return synth.frozen_mask(N, K, design_db)


def _code(case):
    """The code's handle with its decoder compiled for this batch size (kept, as a program
    keeps it for every frame it decodes)."""
    key = tuple(case[k] for k in ("N", "K", "design_db", "frames", "dtype", "compiled"))
    if key not in _codes:
        N, K, frames, dtype = case["N"], case["K"], case["frames"], case["dtype"]
        mask = _mask(N, K, case["design_db"])
        code = polar.polar_code_create(N, K, mask)
        if case["compiled"]:
            shape, _ = autotune.shape_for(N, K, mask, dtype, latency=frames <= 4)
            autotune.configure(code, dtype, shape, frames)
        _codes[key] = code
    return _codes[key]


def _batch(dtype):
    if dtype not in _batches:
        codes = [polar.polar_code_create(N, K, _mask(N, K, synth.MIXED_DESIGN_DB))
                 for N, K in synth.MIXED_CODES]
        shape, _ = autotune.batch_shape(dtype)
        _batches[dtype] = polar.polar_batch_create(codes, dtype == "i8", **shape)
    return _batches[dtype]


# ---------------------------------------------------------------- inputs

def _transform(x):
    """x F^{(x)n} on rows of 0/1 values (natural order), in place."""
    n, N = x.shape
    h = 1
    while h < N:
        v = x.view(n, N // (2 * h), 2, h)
        v[:, :, 0] ^= v[:, :, 1]
        h *= 2
    return x


def _encode(bits, frozen):
    """Systematic codewords (0/1, [n, N]) of information bits [n, K]: transform, clear the
    frozen positions, transform."""
    info = torch.as_tensor(np.flatnonzero(frozen == 0), device=bits.device)
    x = torch.zeros((bits.shape[0], frozen.size), dtype=torch.uint8, device=bits.device)
    x[:, info] = bits
    x = _transform(x)
    x *= torch.as_tensor(1 - frozen, dtype=torch.uint8, device=bits.device)
    return _transform(x)


def _llrs(N, K, frozen, frames, dtype, ebn0_db, gen):
    """Random codewords through BPSK-AWGN, [frames, N] on the device."""
    out = torch.empty((frames, N), dtype=torch.int8 if dtype == "i8" else torch.float32, device=DEV)
    s2 = synth.sigma2(ebn0_db, K / N)
    step = max(1, (1 << 26) // N)
    for f in range(0, frames, step):
        n = min(step, frames - f)
        bits = torch.randint(0, 2, (n, K), generator=gen, device=DEV, dtype=torch.uint8)
        y = torch.randn((n, N), generator=gen, device=DEV)
        y.mul_(s2 ** 0.5).add_(1.0 - 2.0 * _encode(bits, frozen)).mul_(2.0 / s2)
        out[f:f + n] = y.mul_(8.0).round_().clamp_(-127, 127) if dtype == "i8" else y
    return out


def _prepare_mixed(case, gen):
    batch, n = _batch(case["dtype"]), case["frames"]
    share = len(synth.MIXED_CODES)  # equal shares of the codes, as a uniform draw gives
    order = sorted(range(len(synth.MIXED_CODES)), key=lambda c: -synth.MIXED_CODES[c][0])
    parts, ids, lo, oo = [], [], [], []
    pos = opos = 0
    for c in order:  # longest code first, the order a batch is claimed in
        N, K = synth.MIXED_CODES[c]
        m, row = n // share + (c < n % share), (K + 7) // 8
        parts.append(_llrs(N, K, batch.codes[c].frozen, m, case["dtype"], case["ebn0_db"], gen).view(-1))
        ids.append(np.full(m, c, np.int32))
        lo.append(pos + N * np.arange(m, dtype=np.int64))
        oo.append(opos + row * np.arange(m, dtype=np.int64))
        pos, opos = pos + N * m, opos + row * m
    dev = lambda a: torch.as_tensor(np.concatenate(a), device=DEV)  # noqa: E731
    return dict(case=case, batch=batch, ids=dev(ids), lo=dev(lo), oo=dev(oo), llr=torch.cat(parts),
                out=torch.zeros(opos, dtype=torch.uint8, device=DEV))


def prepare(case, seed):
    gen = torch.Generator(device=DEV).manual_seed(int(seed))
    if case["path"] == "mixed":
        return _prepare_mixed(case, gen)
    N, K, n = case["N"], case["K"], case["frames"]
    code = _code(case)
    row, dt = (K + 7) // 8, torch.int8 if case["dtype"] == "i8" else torch.float32
    if case["path"] == "sim":
        u8 = lambda r: torch.zeros((n, r), dtype=torch.uint8, device=DEV)  # noqa: E731
        return dict(case=case, code=code, seed=int(seed), info=u8(row), cw=u8((N + 7) // 8),
                    llr=torch.zeros((n, N), dtype=dt, device=DEV), out=u8(row),
                    errors=torch.zeros(2, dtype=torch.int64, device=DEV))
    llr = _llrs(N, K, code.frozen, n, case["dtype"], case["ebn0_db"], gen)
    if case["path"] == "host":
        llr = llr.cpu().pin_memory()
        out = torch.zeros((n, row), dtype=torch.uint8).pin_memory()
    else:
        out = torch.zeros((n, row), dtype=torch.uint8, device=DEV)
    return dict(case=case, code=code, llr=llr, out=out)


# ---------------------------------------------------------------- one pass

def run(state):
    s, case = state, state["case"]
    if case["path"] == "mixed":
        return polar.polar_batch_decode(s["batch"], s["ids"], s["lo"], s["oo"], s["llr"], s["out"])
    if case["path"] == "host":
        return polar.polar_decode_host(s["code"], s["llr"], s["out"])
    decode = polar.polar_decode_i8 if case["dtype"] == "i8" else polar.polar_decode
    if case["path"] == "decode":
        return decode(s["code"], s["llr"], s["out"])
    polar.polar_random_info(s["code"], s["info"], s["seed"])
    polar.polar_encode_systematic_device(s["code"], s["info"], s["cw"])
    polar.polar_channel_awgn(s["code"], s["cw"], s["llr"], case["ebn0_db"], s["seed"])
    decode(s["code"], s["llr"], s["out"])
    s["errors"].zero_()
    polar.polar_count_errors(s["code"], s["out"], s["info"], s["errors"])
    return {"info": s["info"], "codewords": s["cw"], "llr": s["llr"], "decoded": s["out"],
            "errors": s["errors"]}


# ---------------------------------------------------------------- what a pass cannot do without

def _element_ops(frozen):
    """Element operations of the Fast-SSC tree (Listing 1's calls): N_v / 2 for each F, G and
    Combine, N_v for each constituent decoder."""
    pre = np.concatenate([[0], np.cumsum(frozen, dtype=np.int64)])
    ops, stack = 0, [(0, len(frozen))]
    while stack:
        off, n = stack.pop()
        nf = int(pre[off + n] - pre[off])
        if nf == n:
            continue
        if nf == 0 or (nf == n - 1 and not frozen[off + n - 1]) or (nf == 1 and frozen[off]):
            ops += n
            continue
        h = n // 2
        left0 = int(pre[off + h] - pre[off]) == h
        ops += h if left0 else n      # G_0R alone, or F and G
        ops += h                      # Combine
        stack += [(off + h, h)] if left0 else [(off, h), (off + h, h)]
    return ops


def _decode_work(N, K, frozen, frames, dtype):
    return frames * (N * (1 if dtype == "i8" else 4) + (K + 7) // 8), frames * _element_ops(frozen)


def work(case):
    if case["path"] == "mixed":
        by = ops = 0
        share = case["frames"] / len(synth.MIXED_CODES)
        for N, K in synth.MIXED_CODES:
            b, o = _decode_work(N, K, _mask(N, K, synth.MIXED_DESIGN_DB), 1, case["dtype"])
            by, ops = by + share * b, ops + share * o
        return {"bytes": int(by) + 20 * case["frames"], "flops": int(ops)}
    N, K, n = case["N"], case["K"], case["frames"]
    by, ops = _decode_work(N, K, _mask(N, K, case["design_db"]), n, case["dtype"])
    if case["path"] == "sim":  # bits, codewords, LLRs and decoded bits are each written once
        by += n * ((N + 7) // 8 + (K + 7) // 8)
        ops += n * N * 45          # Philox and Box-Muller per channel value
    return {"bytes": by, "flops": ops}


# ---------------------------------------------------------------- the same in 64 bits

def _philox(c0, c1, c2, c3, seed):
    """Philox-4x32-10 on int64 tensors holding 32-bit words."""
    m = 0xFFFFFFFF
    k0, k1 = seed & m, (seed >> 32) & m
    for r in range(10):
        if r:
            k0, k1 = (k0 + 0x9E3779B9) & m, (k1 + 0xBB67AE85) & m
        p0, p1 = c0 * 0xD2511F53, c2 * 0xCD9E8D57
        c0, c1, c2, c3 = ((p1 >> 32) & m) ^ c1 ^ k0, p1 & m, ((p0 >> 32) & m) ^ c3 ^ k1, p0 & m
    return c0, c1, c2, c3


def exact(case, seed):
    """The channel LLRs of a float32 simulation in 64 bits; every other output is bits."""
    if case["path"] != "sim" or case["dtype"] != "f32":
        return None
    N, K, n, seed = case["N"], case["K"], case["frames"], int(seed)
    frozen = _mask(N, K, case["design_db"])
    s2 = synth.sigma2(case["ebn0_db"], K / N)
    llr = torch.empty((n, N), dtype=torch.float64, device=DEV)
    step = max(1, (1 << 22) // N)
    for f in range(0, n, step):
        m = min(step, n - f)
        fr = torch.arange(f, f + m, device=DEV, dtype=torch.int64)[:, None]

        def words(count, stream):
            j = torch.arange(count, device=DEV, dtype=torch.int64)[None, :] + 0 * fr
            return _philox(j, fr + 0 * j, torch.zeros_like(j), torch.full_like(j, stream), seed)

        w = torch.stack(words((K + 127) // 128, 1), dim=2).reshape(m, -1)
        k = torch.arange(K, device=DEV)
        bits = ((w[:, k // 32] >> (k % 32)) & 1).to(torch.uint8)
        x = _encode(bits, frozen)
        r = [v.double() for v in words((N + 3) // 4, 2)]
        a = [torch.sqrt(-2.0 * torch.log((r[i] + 1.0) * 2.0 ** -32)) for i in (0, 2)]
        t = [2.0 * math.pi * r[i] * 2.0 ** -32 for i in (1, 3)]
        z = torch.stack([a[0] * torch.cos(t[0]), a[0] * torch.sin(t[0]),
                         a[1] * torch.cos(t[1]), a[1] * torch.sin(t[1])], dim=2).reshape(m, -1)
        llr[f:f + m] = (2.0 / s2) * ((1.0 - 2.0 * x.double()) + math.sqrt(s2) * z[:, :N])
    return {"info": None, "codewords": None, "llr": llr, "decoded": None, "errors": None}
