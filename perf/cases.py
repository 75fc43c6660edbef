"""Workloads of the TurboAngle codec: what a program that keeps its KV cache as
records asks of it, through the package's public calls.

A case names one call: `op` (what it does), the cache's shape, its codebooks and
how it is called.

  encode   prefill: rows of every (layer, K/V) block -> records
  append   one decode step: one token per sequence, rows -> record slots of paged pools
  decode   records -> rows, whole blocks
  gather   records -> rows through a slot table (paged pools)
  attend   attention of a GQA group's queries straight from the records

`call` is the entry point: "block" (tac.encode / tac.decode on one block),
"direct" (one batched call, its job array marshalled every time: activations in
new buffers) or "prepared" (the array marshalled once: buffers that stay).
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2603_27467_gb300 as tac

PAGE = 16          # tokens per page of a paged pool
ROUND = 256        # capacity of a contiguous cache: a multiple of this

# (bits, mode) of the K and V norms
NORMS = {
    "k8v4log": ((8, tac.NORM_LINEAR), (4, tac.NORM_LOG)),     # the default scheme
    "norm8": ((8, tac.NORM_LINEAR), (8, tac.NORM_LINEAR)),
    "fp32": ((32, tac.NORM_FP32), (32, tac.NORM_FP32)),       # angle-only
}


def _case(name, op, call, layers, heads, d, tokens, *, seqs=1, kv="both", dtype="bf16", n_k=64, n_v=64, n_early=256,
          norms="k8v4log", nq=0, tokens_lo=0):
    return dict(name=name, op=op, call=call, layers=layers, heads=heads, d=d, tokens=tokens, seqs=seqs, kv=kv,
                dtype=dtype, n_k=n_k, n_v=n_v, n_early=n_early, norms=norms, nq=nq, tokens_lo=tokens_lo)


def listed():
    return [
        # one K block of a short prompt, the smallest call: its latency is launches and host work
        _case("encode_block_short", "encode", "block", 1, 8, 128, 33, kv="k"),
        # one layer's K block read back in fp32, head dimension 64
        _case("decode_block_1k", "decode", "block", 1, 8, 64, 1024, kv="k", dtype="fp32"),
        # a decode step of a single conversation: 8 rows for each of 64 caches, scattered
        _case("append_1seq", "append", "prepared", 32, 8, 128, 1, seqs=1),
        # a decode step of a serving batch
        _case("append_256seq", "append", "prepared", 32, 8, 128, 1, seqs=256),
        # prefill of an odd-length prompt on a small model (d = 64): activations in new buffers
        _case("encode_prompt_d64", "encode", "direct", 16, 8, 64, 2047, n_k=128, n_v=64),
        # angle-only records (fp32 norms) with a codebook that is no power of two
        _case("encode_fp32norm_n56", "encode", "prepared", 22, 4, 64, 8191, n_k=56, n_v=56, n_early=0, norms="fp32"),
        # a whole 32k-token cache of a 7B model, in and out: the largest calls
        _case("encode_cache_32k", "encode", "prepared", 32, 8, 128, 32768),
        _case("decode_cache_32k", "decode", "prepared", 32, 8, 128, 32768),
        # four sequences read back from paged pools (swap-out, migration to another engine)
        _case("gather_paged_d64", "gather", "prepared", 16, 8, 64, 3001, seqs=4, n_k=128, n_v=64),
        # attention of one layer of one conversation, as a decode step makes it layer by layer
        _case("attend_layer_4k", "attend", "prepared", 1, 8, 128, 4097, nq=4, n_early=0),
        # the same for a batch of sequences of very different lengths
        _case("attend_batch_ragged", "attend", "prepared", 1, 8, 128, 32768, seqs=16, tokens_lo=1024, nq=4, n_early=0),
        # a small model's whole step (d = 64), fp32 queries
        _case("attend_step_d64", "attend", "prepared", 16, 8, 64, 8192, nq=4, dtype="fp32", n_k=128, n_v=64),
    ]


def _log(rng, lo, hi):
    """A whole number spread over the logarithm of [lo, hi], odd as often as not."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    op = rng.choice(["encode", "encode", "append", "decode", "gather", "attend", "attend"])
    d = rng.choice([64, 128, 128])
    heads = rng.choice([4, 8])
    norms = rng.choice(["k8v4log", "k8v4log", "norm8", "fp32"])
    ns = [16, 32, 48, 56, 64, 64, 128, 256]
    c = dict(op=op, call="prepared", layers=_log(rng, 1, 32), heads=heads, d=d, tokens=1, seqs=1, kv="both",
             dtype=rng.choice(["bf16", "bf16", "fp32"]), n_k=rng.choice(ns), n_v=rng.choice(ns),
             n_early=rng.choice([0, 256]), norms=norms, nq=0, tokens_lo=0)
    # rows of a block are bounded so that no draw is larger than a 32k-token cache of 32 layers x 8 heads
    cap = 32768 * 32 * 8
    if op == "append":
        c["seqs"] = _log(rng, 1, 256)
    elif op == "attend":
        c["layers"] = rng.choice([1, 1, c["layers"]])
        c["seqs"] = _log(rng, 1, max(1, min(32, 160 // c["layers"])))
        c["nq"] = rng.choice([1, 2, 4, 4, 8])
        c["tokens"] = _log(rng, 1, max(64, min(32768, cap // (2 * c["layers"] * heads * c["seqs"]))))
        c["tokens_lo"] = rng.choice([0, max(1, c["tokens"] // 16)])
    else:
        c["call"] = rng.choice(["block", "direct", "prepared"]) if op != "gather" else rng.choice(["direct", "prepared"])
        if c["call"] == "block":
            c["layers"], c["kv"] = 1, rng.choice(["k", "v"])
        if op == "gather":
            c["seqs"] = _log(rng, 1, 16)
        c["tokens"] = _log(rng, 1, min(32768, cap // (2 * c["layers"] * heads * c["seqs"])))
    return c


# ---------------------------------------------------------------------------
# shapes
# ---------------------------------------------------------------------------
def _blocks(c):
    """(layer, kv, n, bits, mode) of every (layer, K/V) cache."""
    out = []
    for layer in range(c["layers"]):
        for kv, name in ((0, "k"), (1, "v")):
            if c["kv"] not in ("both", name):
                continue
            n = c["n_early"] if c["n_early"] and layer < 4 and c["layers"] > 1 else (c["n_k"], c["n_v"])[kv]
            bits, mode = NORMS[c["norms"]][kv]
            out.append((layer, kv, n, bits, mode))
    return out


def _lengths(c):
    """Tokens of each sequence: spread over the logarithm of [tokens_lo, tokens], or all `tokens`."""
    lo, hi, s = c["tokens_lo"], c["tokens"], c["seqs"]
    if not lo:
        return [hi] * s
    return [max(1, int(lo * (hi / lo) ** ((i + 0.5) / s))) | (i & 1) for i in range(s)]


def _rows(c):
    """Rows of one block."""
    return c["heads"] * sum(_lengths(c))


def _code_bits(n):
    return max(1, math.ceil(math.log2(n)))


def _row_bytes(c, n, bits, mode):
    p = c["d"] // 2
    return p * _code_bits(n) // 8 + p * bits // 8 + (0 if mode == tac.NORM_FP32 else 8)


def _dtype(c):
    return torch.bfloat16 if c["dtype"] == "bf16" else torch.float32


def work(c):
    d, esz = c["d"], 2 if c["dtype"] == "bf16" else 4
    rows = _rows(c)
    total, flops = 0.0, 0.0
    for _, _, n, bits, mode in _blocks(c):
        if c["op"] == "attend":
            total += rows * _row_bytes(c, n, bits, mode)
        else:
            total += rows * (d * esz + _row_bytes(c, n, bits, mode) + (8 if c["op"] in ("append", "gather") else 0))
        # the transform's additions, or one multiply-add per query, and about ten operations a pair
        flops += rows * (2 * d * c["nq"] if c["op"] == "attend" else d * math.log2(d)) + rows * (d // 2) * 10
    if c["op"] == "attend":
        total += 2 * c["layers"] * c["seqs"] * c["heads"] * c["nq"] * d * esz   # queries and outputs
    return {"bytes": total, "flops": flops}


def tolerance(c):
    if c["op"] in ("encode", "append"):
        # codes are bytes and stay the same; the header's (r_min, r_max) and the fp32 norms are fp32
        # results of a fp32 transform
        return {"rel": 2e-7, "max": 4e-6}      # 5e-8 from 64 bits
    if c["dtype"] == "bf16":
        return {"rel": 6e-3, "max": 2e-2}      # one rounding to bf16: 1.7e-3 from 64 bits
    if c["op"] == "attend":
        return {"rel": 2.5e-6, "max": 2.5e-5}  # fp32 scores and softmax sums: 6e-7 from 64 bits
    return {"rel": 5e-7, "max": 1e-5}          # fp32 transform, hardware ex2 / lg2 of log-space norms: 1e-7 from 64 bits


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _gen(seed, *key):
    g = torch.Generator(device="cuda")
    v = int(seed) & 0x7FFFFFFF
    for k in key:
        v = (v * 1_000_003 + int(k) + 1) & 0x7FFFFFFFFFFF
    g.manual_seed(v)
    return g


def _values(c, rows_per_head, layer, kv, seed):
    """Rows [heads * rows_per_head, d] with channel scales (lognormal, 1-2 % outlier channels) and a scale per token."""
    g = _gen(seed, 11, layer, kv)
    h, d = c["heads"], c["d"]
    s, m, t = (1.0, 20.0, 0.0) if d == 128 else (0.5, 10.0, 0.3)
    sigma = torch.exp(s * torch.randn((h, 1, d), generator=g, device="cuda"))
    out = torch.randint(0, d, (h, 1, 1), generator=g, device="cuda")
    sigma.scatter_(2, out, sigma.gather(2, out) * m)
    x = torch.randn((h, rows_per_head, d), generator=g, device="cuda")
    x *= sigma
    if t:
        x *= torch.exp(t * torch.randn((1, rows_per_head, 1), generator=g, device="cuda"))
    return x.to(_dtype(c)).reshape(h * rows_per_head, d)


def _pack6(k):
    """Codes < 64 in 6-bit fields, LSB first."""
    k = k.reshape(k.shape[0], -1, 4).to(torch.int32)
    w = k[..., 0] | (k[..., 1] << 6) | (k[..., 2] << 12) | (k[..., 3] << 18)
    return torch.stack([w & 255, (w >> 8) & 255, w >> 16], dim=-1).to(torch.uint8).reshape(k.shape[0], -1)


def _records(c, slots, n, bits, mode, codes, norms, off, layer, kv, seq, seed):
    """Fills one cache's planes (`slots` records) with records as encoding leaves them: angle codes
    uniform over the bins, norm codes of Rayleigh norms against the row's extremes, their header."""
    g = _gen(seed, 23, layer, kv, seq)
    p = c["d"] // 2
    ab, nb = p * _code_bits(n) // 8, p * bits // 8
    if n & (n - 1):
        codes[: slots * ab] = _pack6(torch.randint(0, n, (slots, p), generator=g, device="cuda", dtype=torch.uint8)).reshape(-1)
    else:
        codes[: slots * ab] = torch.randint(0, 256, (slots * ab,), generator=g, device="cuda", dtype=torch.uint8)
    r = torch.sqrt(torch.empty((slots, p), device="cuda").exponential_(0.5, generator=g))   # |(N(0,1), N(0,1))|
    r *= torch.exp(0.25 * torch.randn((slots, 1), generator=g, device="cuda"))
    if mode == tac.NORM_FP32:
        norms[: slots * nb] = r.view(torch.uint8).reshape(-1)
        return
    lo, hi = r.amin(dim=1, keepdim=True), r.amax(dim=1, keepdim=True)
    top = (1 << bits) - 1
    f = torch.log2 if mode == tac.NORM_LOG else (lambda v: v)
    q = torch.floor((f(r) - f(lo)) / (f(hi) - f(lo)) * top + 0.5).clamp_(0, top).to(torch.uint8)
    if bits == 4:
        q = q[:, 0::2] | (q[:, 1::2] << 4)
    norms[: slots * nb] = q.reshape(-1)
    norms[off: off + 8 * slots] = torch.cat([lo, hi], dim=1).view(torch.uint8).reshape(-1)


def _up16(v):
    return (v + 15) // 16 * 16


class _Planes:
    """Record planes of all caches of one codebook in two buffers, a row for each cache."""

    def __init__(self, c, count, capacity, n, bits, mode):
        self.mode, self.capacity = mode, capacity
        cfg = tac.layer_cfg(c["d"], n, bits, mode)
        self.cb, self.nb = tac.codes_bytes(cfg, capacity), capacity * tac.norm_row_bytes(cfg)
        self.off = tac.header_offset(cfg, capacity)
        self.codes = torch.zeros((count, _up16(self.cb)), dtype=torch.uint8, device="cuda")
        self.norms = torch.zeros((count, _up16(tac.norms_bytes(cfg, capacity))), dtype=torch.uint8, device="cuda")

    def out(self):
        if self.mode == tac.NORM_FP32:
            return {"angle": self.codes[:, : self.cb], "norm": self.norms[:, : self.nb].view(torch.float32)}
        return {"angle": self.codes[:, : self.cb], "norm": self.norms[:, : self.nb],
                "header": self.norms[:, self.off: self.off + 8 * self.capacity].view(torch.float32)}


def _pools(c, capacity):
    """One cache per block: ({(n, bits, mode): planes}, caches in block order)."""
    planes, at, caches = {}, {}, []
    blocks = _blocks(c)
    for _, _, n, bits, mode in blocks:
        at[(n, bits, mode)] = at.get((n, bits, mode), 0) + 1
    for key, count in at.items():
        planes[key] = _Planes(c, count, capacity, *key)
    at = dict.fromkeys(at, 0)
    for layer, kv, n, bits, mode in blocks:
        pl, i = planes[(n, bits, mode)], at[(n, bits, mode)]
        at[(n, bits, mode)] = i + 1
        cfg = tac.layer_cfg(c["d"], n, bits, mode, 0, layer, kv)
        caches.append(tac.Cache(cfg, capacity, pl.codes[i], pl.norms[i]))
    return planes, caches


def _paged_slots(c, seed):
    """(record slots int64, pool capacity): for append the last token of each sequence (row = sequence, head),
    for gather every token (row = sequence, head, token); pages in random order, a page holds PAGE tokens of each head."""
    g = np.random.default_rng([int(seed) & 0xFFFFFFFF, 31])
    h = np.arange(c["heads"])
    if c["op"] == "append":
        pages = g.permutation(c["seqs"] + 3)[: c["seqs"]]
        pos = g.integers(0, PAGE, c["seqs"])
        s = (pages[:, None] * c["heads"] + h[None, :]) * PAGE + pos[:, None]
        total = c["seqs"] + 3
    else:
        per = -(-c["tokens"] // PAGE)
        total = c["seqs"] * per + 3
        pages = g.permutation(total)[: c["seqs"] * per].reshape(c["seqs"], 1, per)
        t = np.arange(c["tokens"])
        s = (pages[:, :, t // PAGE] * c["heads"] + h[None, :, None]) * PAGE + (t % PAGE)[None, None, :]
    return torch.from_numpy(s.reshape(-1).astype(np.int64)).cuda(), total * c["heads"] * PAGE


def prepare(c, seed):
    blocks, d = _blocks(c), c["d"]
    if c["op"] in ("encode", "append"):
        slot, capacity = _paged_slots(c, seed) if c["op"] == "append" else (None, _rows(c))
        planes, caches = _pools(c, capacity)
        x = [_values(c, c["seqs"] * c["tokens"], layer, kv, seed) for layer, kv, *_ in blocks]
        if c["call"] == "block":
            return {"call": lambda: tac.encode(x[0], caches[0].cfg, caches[0]), "out": [p.out() for p in planes.values()]}
        jobs = [tac.EncodeJob(ca.cfg, xi, ca, slot) for ca, xi in zip(caches, x)]
        call = tac.encode_multi_prepared(jobs) if c["call"] == "prepared" else (lambda: tac.encode_multi(jobs))
        return {"call": call, "out": [p.out() for p in planes.values()]}
    if c["op"] in ("decode", "gather"):
        slot, capacity = _paged_slots(c, seed) if c["op"] == "gather" else (None, _rows(c))
        planes, caches = _pools(c, capacity)
        for ca, (layer, kv, n, bits, mode) in zip(caches, blocks):
            _records(c, capacity, n, bits, mode, ca.codes, ca.norms, tac.header_offset(ca.cfg, capacity), layer, kv, 0, seed)
        y = torch.zeros((len(blocks), _rows(c), d), dtype=_dtype(c), device="cuda")
        if c["call"] == "block":
            return {"call": lambda: tac.decode(caches[0], caches[0].cfg, y=y[0]), "out": y}
        jobs = [tac.DecodeJob(ca.cfg, ca, y[i], slot) for i, ca in enumerate(caches)]
        call = tac.decode_multi_prepared(jobs) if c["call"] == "prepared" else (lambda: tac.decode_multi(jobs))
        return {"call": call, "out": y}
    # attend: a cache for each (layer, sequence, KV head)
    q = _queries(c, seed)
    out = torch.zeros_like(q)
    jobs = []
    for layer in range(c["layers"]):
        two = [b for b in blocks if b[0] == layer]
        for s, length in enumerate(_lengths(c)):
            capacity = -(-length // ROUND) * ROUND
            kv = []
            for _, which, n, bits, mode in two:
                pl = _Planes(c, c["heads"], capacity, n, bits, mode)
                cfg = tac.layer_cfg(d, n, bits, mode, 0, layer, which)
                for h in range(c["heads"]):
                    _records(c, capacity, n, bits, mode, pl.codes[h], pl.norms[h], pl.off, layer, which,
                             s * c["heads"] + h, seed)
                kv.append([tac.Cache(cfg, capacity, pl.codes[h], pl.norms[h]) for h in range(c["heads"])])
            for h in range(c["heads"]):
                k, v = kv[0][h], kv[1][h]
                jobs.append(tac.AttendJob(k.cfg, k, v.cfg, v, length, q[layer, s, h], out[layer, s, h], 1.0 / math.sqrt(d)))
    return {"call": tac.attend_multi_prepared(jobs), "out": out}


def _queries(c, seed):
    q = 2.0 * torch.randn((c["layers"], c["seqs"], c["heads"], c["nq"], c["d"]), generator=_gen(seed, 41), device="cuda")
    return q.to(_dtype(c))


def run(state):
    state["call"]()
    return state["out"]


# ---------------------------------------------------------------------------
# the same in 64 bits
# ---------------------------------------------------------------------------
def _mix(z, i):
    m = (1 << 64) - 1
    z = (z + (i + 1) * 0x9E3779B97F4A7C15) & m
    z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & m
    z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & m
    return z ^ (z >> 31)


def _signs64(d, layer, kv):
    """The +-1 diagonal of (layer, K/V), seed 0: SplitMix64 streams."""
    key = _mix(0, 2 * layer + kv)
    return torch.tensor([-1.0 if _mix(key, j) >> 63 else 1.0 for j in range(d)], dtype=torch.float64, device="cuda")


def _hadamard64(d):
    h = torch.ones((1, 1), dtype=torch.float64, device="cuda")
    while h.shape[0] < d:
        h = torch.cat([torch.cat([h, h], 1), torch.cat([h, -h], 1)], 0)
    return h / math.sqrt(d)


def _order(d):
    """The pair whose code is in position v of a record."""
    p = d // 2
    if d not in (64, 128):
        return torch.arange(p, device="cuda")
    m = d // 16
    return torch.tensor([4 * (v % m) + (v // m) % 4 + 4 * m * (v // (4 * m)) for v in range(p)], device="cuda")


def _fields(plane, w):
    """Codes of w bits, LSB first, from a byte plane [rows, bytes]."""
    if w == 8:
        return plane
    if w == 6:
        b = plane.reshape(plane.shape[0], -1, 3).to(torch.int32)
        v = b[..., 0] | (b[..., 1] << 8) | (b[..., 2] << 16)
        return torch.stack([(v >> (6 * j)) & 63 for j in range(4)], dim=-1).reshape(plane.shape[0], -1)
    b = plane.reshape(plane.shape[0], -1, w).to(torch.int64)     # w bytes hold 8 codes
    v = sum(b[..., j] << (8 * j) for j in range(w))
    return torch.stack([(v >> (w * j)) & ((1 << w) - 1) for j in range(8)], dim=-1).reshape(plane.shape[0], -1)


def _pairs64(c, slots, n, bits, mode, layer, kv, seq, seed):
    """The rotated rows y^ [slots, d] that one cache's records stand for, in 64 bits."""
    d, p = c["d"], c["d"] // 2
    w = _code_bits(n)
    codes = torch.zeros(slots * p * w // 8, dtype=torch.uint8, device="cuda")
    off = _up16(slots * p * bits // 8)
    norms = torch.zeros(off + 8 * slots, dtype=torch.uint8, device="cuda")
    _records(c, slots, n, bits, mode, codes, norms, off, layer, kv, seq, seed)
    k = _fields(codes.reshape(slots, -1), w).to(torch.float64)
    if mode == tac.NORM_FP32:
        r = norms[: slots * p * 4].view(torch.float32).reshape(slots, p).to(torch.float64)
    else:
        v = _fields(norms[: slots * p * bits // 8].reshape(slots, -1), bits).to(torch.float64)
        hd = norms[off:].view(torch.float32).reshape(slots, 2).to(torch.float64)
        lo, hi = hd[:, :1], hd[:, 1:]
        top = (1 << bits) - 1
        if mode == tac.NORM_LOG:
            r = torch.exp2(torch.log2(lo) + v * (torch.log2(hi) - torch.log2(lo)) / top)
        else:
            r = lo + v * (hi - lo) / top
    a = k * (2.0 * math.pi / n)
    y = torch.empty((slots, p, 2), dtype=torch.float64, device="cuda")
    order = _order(d)
    y[:, order, 0] = r * torch.cos(a)
    y[:, order, 1] = r * torch.sin(a)
    return y.reshape(slots, d)


def exact(c, seed):
    blocks, d = _blocks(c), c["d"]
    h64 = _hadamard64(d)
    if c["op"] in ("encode", "append"):
        # the header (or the fp32 norms); the codes are bytes and have no 64-bit value
        slot, capacity = _paged_slots(c, seed) if c["op"] == "append" else (None, _rows(c))
        order = _order(d)
        got = {}
        for layer, kv, n, bits, mode in blocks:
            x = _values(c, c["seqs"] * c["tokens"], layer, kv, seed).to(torch.float64)
            y = ((x * _signs64(d, layer, kv)) @ h64).reshape(-1, d // 2, 2)
            r = torch.hypot(y[..., 0], y[..., 1])
            if mode == tac.NORM_FP32:
                v = r[:, order]
            else:
                lo, hi = r.amin(dim=1), r.amax(dim=1)
                v = torch.stack([torch.maximum(lo, hi * 2.0**-24) if mode == tac.NORM_LOG else lo, hi], dim=1)
            if slot is not None:
                full = torch.zeros((capacity, v.shape[1]), dtype=torch.float64, device="cuda")
                full[slot] = v
                v = full
            got.setdefault((n, bits, mode), []).append(v.reshape(-1))
        return [{"angle": None, "norm": torch.stack(v)} if key[2] == tac.NORM_FP32 else
                {"angle": None, "norm": None, "header": torch.stack(v)} for key, v in got.items()]
    if c["op"] in ("decode", "gather"):
        slot, capacity = _paged_slots(c, seed) if c["op"] == "gather" else (None, _rows(c))
        out = torch.empty((len(blocks), _rows(c), d), dtype=torch.float64, device="cuda")
        for i, (layer, kv, n, bits, mode) in enumerate(blocks):
            y = _pairs64(c, capacity, n, bits, mode, layer, kv, 0, seed)
            if slot is not None:
                y = y[slot]
            out[i] = (y @ h64) * _signs64(d, layer, kv)
        return out
    q = _queries(c, seed).to(torch.float64)
    out = torch.empty_like(q)
    for layer in range(c["layers"]):
        (_, _, nk, bk, mk), (_, _, nv, bv, mv) = [b for b in blocks if b[0] == layer]
        dk, dv = _signs64(d, layer, 0), _signs64(d, layer, 1)
        for s, length in enumerate(_lengths(c)):
            capacity = -(-length // ROUND) * ROUND
            for h in range(c["heads"]):
                at = s * c["heads"] + h
                k = _pairs64(c, capacity, nk, bk, mk, layer, 0, at, seed)[:length]
                v = _pairs64(c, capacity, nv, bv, mv, layer, 1, at, seed)[:length]
                w = torch.softmax(((q[layer, s, h] * dk) @ h64) @ k.T / math.sqrt(d), dim=-1)
                out[layer, s, h] = ((w @ v) @ h64) * dv
    return out
