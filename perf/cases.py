"""What a program that keeps a bounded KV cache has this library do, as timed cases.

Every case is one turn of such a program through the public binding, at the shapes of the
repository's own workloads (``synth.WORKLOADS``) or generic ones:

  cycle    a full cache is compressed in place and the next chunk of rows is appended, which fills
           it again -- the chunk-wise loop of prefilling and the event of a decode stream;
  ragged   a batch of caches of different lengths is compressed in one call;
  decode   one token per sequence: its rows are appended for all layers, then every layer attends;
  prefill  one chunk per sequence: its rows are appended for all layers, then every layer attends.

Inputs are AR(1) sequences with outlier channels, the library's stand-in for real key/value states.
"""
from __future__ import annotations

import math

import torch

from paper_2505_00570_b200 import binding as fk
from paper_2505_00570_b200 import synth

DTYPES = {"bf16": torch.bfloat16, "fp32": torch.float32}
SIZES = {"bf16": 2, "fp32": 4}


def _shape(op, batch, layers, kv_heads, head_dim, capacity, dtype="bf16", sink=4, rho=0.9, **more):
    return dict(op=op, batch=batch, layers=layers, kv_heads=kv_heads, head_dim=head_dim, capacity=capacity, dtype=dtype,
                sink=sink, rho=rho, **more)


def listed():
    return [
        # The smallest call there is: one head, a short fp32 cache, no sinks.  Launches and host work.
        dict(_shape("cycle", 1, 1, 1, 128, 512, "fp32", sink=0, kept=256), name="cycle_tiny_fp32"),
        # LLaMA-2-7B shapes, one sequence: the paper's own 4092 -> 2046 of all layers, the headline workload.
        dict(_shape("cycle", 1, 32, 32, 128, 4096, kept=2046), name="cycle_7b"),
        # LLaMA-3-8B shapes, a batch of 8 long caches (8188 -> 4094): the largest call.
        dict(_shape("cycle", 8, 32, 8, 128, 8192, rho=0.95, kept=4094), name="cycle_8b"),
        # A retaining ratio of one quarter on a cache of odd length (2997 -> 749), GQA heads.
        dict(_shape("cycle", 4, 32, 8, 128, 3001, kept=749), name="cycle_quarter_odd"),
        # A model with heads of 64 channels, two sequences, 12 heads in each of 12 layers.
        dict(_shape("cycle", 2, 12, 12, 64, 4096, kept=2046), name="cycle_head64"),
        # An fp32 cache whose lengths are no powers of two (2044 -> 1022).
        dict(_shape("cycle", 1, 4, 8, 128, 2048, "fp32", kept=1022), name="cycle_fp32"),
        # Independent sequences of a serving batch, each with a length of its own, each halved.
        dict(_shape("ragged", 8, 32, 8, 128, 8192, lens="1187 8192 4801 2310 6733 3594 7451 5602"), name="ragged_8b"),
        # One decode step of a batch of 16 on LLaMA-2-7B shapes (multi-head attention), caches nearly full.
        dict(_shape("decode", 16, 4, 32, 128, 4096, group=1, lens="4096"), name="decode_7b"),
        # One decode step of a batch of 8 on LLaMA-3-8B shapes (4 query heads per KV head), long caches.
        dict(_shape("decode", 8, 8, 8, 128, 8192, rho=0.95, group=4, lens="8192 7001 6113 5120 8000 4099 7777 6655"),
             name="decode_8b"),
        # One decode step of a single user: all layers, a cache that was compressed a while ago.
        dict(_shape("decode", 1, 32, 8, 128, 4096, group=4, lens="2611"), name="decode_single"),
        # A prefill chunk on LLaMA-2-7B shapes: the 2046 rows that fill the cache after a compression.
        dict(_shape("prefill", 1, 4, 32, 128, 4096, group=1, n_new=2046, lens="4096"), name="prefill_7b"),
        # A short odd chunk on LLaMA-3-8B shapes for two sequences of different lengths.
        dict(_shape("prefill", 2, 4, 8, 128, 8192, rho=0.95, group=4, n_new=1001, lens="5003 6790"), name="prefill_8b_odd"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["cycle", "cycle", "cycle", "ragged", "decode", "decode", "prefill"])
    kv_heads = rng.choice([4, 8, 8, 32])
    sink = rng.choice([0, 4, 4, 4, rng.randrange(1, 33)])
    rho = rng.choice([0.9, 0.95])
    if op == "cycle":
        dtype, head_dim = rng.choice([("bf16", 128)] * 5 + [("bf16", 64), ("fp32", 128)])
        if dtype == "fp32":
            capacity = _log_int(rng, 256, 4096)
            layers, kv_heads, batch = rng.randrange(1, 5), rng.choice([1, 4, 8]), 1
        elif head_dim == 64:
            capacity = rng.choice([4096, 4000, 2048, 3072, 3200])
            sink = rng.choice([0, 4]) if capacity in (4096, 2048) else 0
            layers, batch = rng.randrange(4, 17), rng.randrange(1, 4)
        else:
            capacity = _log_int(rng, 1024, 8192)
            layers = rng.choice([8, 16, 24, 32, rng.randrange(1, 33)])
            rows = layers * kv_heads * capacity
            batch = max(1, min(8, (32 * 8 * 8192 * 8) // rows, _log_int(rng, 1, 8)))
        ratio = rng.choice([0.5, 0.5, 0.5, 0.25, 0.75]) if head_dim == 128 else 0.5
        kept = int(ratio * (capacity - sink))
        return _shape("cycle", batch, layers, kv_heads, head_dim, capacity, dtype, sink, rho, kept=kept)
    if op == "ragged":
        batch, layers = rng.randrange(2, 9), rng.choice([8, 16, 32])
        kv_heads = min(kv_heads, 8)
        lens = [rng.randrange(1024, 8193) for _ in range(batch)]
        return _shape("ragged", batch, layers, kv_heads, 128, 8192, "bf16", sink, rho, lens=" ".join(map(str, lens)))
    group = 1 if kv_heads == 32 else rng.choice([1, 2, 4, 8])
    capacity = _log_int(rng, 1024, 8192)
    batch = _log_int(rng, 1, 16)
    if op == "decode":
        layers = 4 if kv_heads * batch > 64 else rng.choice([8, 16, 32])
        lens = [rng.randrange(capacity // 3, capacity + 1) for _ in range(batch)]
        return _shape("decode", batch, layers, kv_heads, 128, capacity, "bf16", sink, rho, group=group,
                      lens=" ".join(map(str, lens)))
    batch = min(batch, 4)
    n_new = _log_int(rng, 64, capacity // 2)
    lens = [rng.randrange(max(n_new, capacity // 3), capacity + 1) for _ in range(batch)]
    return _shape("prefill", batch, 2, kv_heads, 128, capacity, "bf16", sink, rho, group=group, n_new=n_new,
                  lens=" ".join(map(str, lens)))


def _lens(case):
    lens = [int(x) for x in case["lens"].split()]
    return lens * case["batch"] if len(lens) == 1 else lens


def _rows(case, n, seed):
    """``n`` consecutive rows of K and of V, dense, drawn on the GPU from the seed."""
    w = synth.Workload("case", case["batch"], case["layers"], case["kv_heads"], case["head_dim"], n, DTYPES[case["dtype"]],
                       case["sink"], case["rho"], 2 if case["dtype"] == "bf16" else 0, seed)
    return synth.make_cache(w, "cuda")


def _inputs(case, seed):
    """The full cache, the rows to append, the lengths and the queries of a case, from the seed alone."""
    st = dict(case=case)
    st["k"], st["v"] = _rows(case, case["capacity"], 10 * seed + 1)
    op = case["op"]
    if op == "cycle":
        n_in = case["capacity"] - case["sink"]
        st["new_k"], st["new_v"] = _rows(case, n_in - case["kept"], 10 * seed + 2)
        st["lens"] = [case["sink"] + case["kept"]] * case["batch"]
        st["pairs"] = [(n_in, case["kept"])] * case["batch"]
    elif op == "ragged":
        st["lens"] = _lens(case)
        st["kept"] = [(n - case["sink"]) // 2 for n in st["lens"]]
        st["pairs"] = [(n - case["sink"], kept) for n, kept in zip(st["lens"], st["kept"])]
    else:
        n_new = case.get("n_new", 1)
        st["new_k"], st["new_v"] = _rows(case, n_new, 10 * seed + 2)
        st["before"] = [n - n_new for n in _lens(case)]
        gen = torch.Generator(device="cuda")
        gen.manual_seed(10 * seed + 3)
        heads = case["kv_heads"] * case["group"]
        size = (case["layers"], case["batch"], heads, case["head_dim"]) if op == "decode" else \
            (case["layers"], case["batch"], heads, n_new, case["head_dim"])
        st["q"] = torch.randn(size, generator=gen, device="cuda").to(DTYPES[case["dtype"]])
        st["pairs"] = []
    return st


def prepare(case, seed):
    st = _inputs(case, seed)
    ctx = st["ctx"] = fk.Context()
    if "q" in st:
        st["out"] = torch.empty_like(st["q"])
    layout = fk.layout_of(st["k"])
    for n_in, kept in dict.fromkeys(st["pairs"]):  # the tables of these lengths, kept by the context
        ctx.plan(n_in, kept, layout.dtype, ctx.resolve_variant(layout, n_in, kept))
    return st


def run(st):
    case, ctx, k, v = st["case"], st["ctx"], st["k"], st["v"]
    op = case["op"]
    if op == "cycle":
        ctx.compress(k, v, case["capacity"], case["kept"], case["sink"])
        ctx.append(k, v, st["new_k"], st["new_v"], st["lens"])
        return k, v
    if op == "ragged":
        ctx.compress_ragged(k, v, st["lens"], st["kept"], case["sink"])
        return k, v
    lens = ctx.append(k, v, st["new_k"], st["new_v"], st["before"])
    attend = ctx.attend_decode if op == "decode" else ctx.attend_prefill
    for layer in range(case["layers"]):
        attend(k, v, layer, st["q"][layer], lens, rope_base=10000.0, out=st["out"][layer])
    return st["out"], k, v


def _transform(n_in, kept):
    # a real transform of n points and one of the kept ones, by the FFT: 2.5 n log2 n each
    return 2.5 * (n_in * math.log2(max(n_in, 2)) + kept * math.log2(max(kept, 2)))


def work(case):
    size, d = SIZES[case["dtype"]], case["head_dim"]
    per_len = 2 * case["layers"] * case["kv_heads"]  # matrices of one sequence, K and V
    row = d * size
    op = case["op"]
    if op == "cycle":
        mats, n_in, kept = per_len * case["batch"], case["capacity"] - case["sink"], case["kept"]
        return dict(bytes=mats * row * (n_in + kept + 2 * (n_in - kept)), flops=mats * d * _transform(n_in, kept))
    if op == "ragged":
        pairs = [(n - case["sink"], (n - case["sink"]) // 2) for n in _lens(case)]
        return dict(bytes=sum(per_len * row * (n + m) for n, m in pairs),
                    flops=sum(per_len * d * _transform(n, m) for n, m in pairs))
    n_new, group = case.get("n_new", 1), case["group"]
    heads = case["layers"] * case["kv_heads"] * group
    append = 2 * per_len * n_new * row * case["batch"]
    io = 2 * heads * n_new * row * case["batch"]
    cached = sum(per_len * n * row for n in _lens(case))
    seen = sum(n_new * (n - n_new) + n_new * (n_new + 1) / 2 for n in _lens(case))  # query, key pairs of one head
    return dict(bytes=append + io + cached, flops=4 * d * heads * seen)


def tolerance(case):
    """Four times the error against the same path in 64 bits: the compression of bf16 caches is 2.5e-3 off (bf16 basis
    and operands, one rounding of the result), the attention 2e-3 (fp16 scores, bf16 weights and result), the
    fp32 compression 4e-7 or less -- but sums of thousands of fp32 terms in another order differ by several times that."""
    return {"rel": 1e-2} if case["dtype"] == "bf16" else {"rel": 5e-6}


def _projection(n_in, kept):
    """The compression of one column as a matrix: sqrt(kept / n_in) * IDCT_kept * (first kept rows of DCT-II_n_in), 64 bits."""
    t = torch.arange(kept, device="cuda")

    def rows(n):  # cos(pi (2 i + 1) t / 2 n), orthonormal, the angle reduced in whole numbers
        i = torch.arange(n, device="cuda")
        c = torch.cos(((2 * i[None, :] + 1) * t[:, None] % (4 * n)).double() * (math.pi / (2 * n))) * math.sqrt(2 / n)
        c[0] *= math.sqrt(0.5)
        return c
    return math.sqrt(kept / n_in) * rows(kept).T @ rows(n_in)


def _rope(x, positions, base=10000.0):
    """Channel c with channel c + d/2, turned by position * base^(-2c/d); x ends in [position, channel]."""
    h = x.shape[-1] // 2
    angle = positions.double()[:, None] * base ** (-torch.arange(h, device="cuda").double() / h)
    cos, sin = torch.cos(angle), torch.sin(angle)
    return torch.cat([x[..., :h] * cos - x[..., h:] * sin, x[..., h:] * cos + x[..., :h] * sin], dim=-1)


def exact(case, seed):
    """What ``run`` returns for these inputs, by plain torch in 64 bits."""
    st = _inputs(case, seed)
    k, v, sink, op = st["k"].double(), st["v"].double(), case["sink"], case["op"]
    for b, (n_in, kept) in enumerate(st["pairs"]):
        p = _projection(n_in, kept)
        for cache in (k, v):
            for layer in range(case["layers"]):
                cache[b, layer, :, sink:sink + kept] = p @ cache[b, layer, :, sink:sink + n_in]
    if op == "ragged":
        return k, v
    for b, at in enumerate(st["lens"] if op == "cycle" else st["before"]):
        for cache, new in ((k, st["new_k"]), (v, st["new_v"])):
            cache[b, :, :, at:at + new.shape[3]] = new[b].double()
    if op == "cycle":
        return k, v
    n_new, group, d = case.get("n_new", 1), case["group"], case["head_dim"]
    q = st["q"].reshape(case["layers"], case["batch"], case["kv_heads"], group, n_new, d)
    out = torch.empty(q.shape, dtype=torch.float64, device="cuda")
    for b, n in enumerate(_lens(case)):
        at = torch.arange(n, device="cuda")
        unseen = at[None, :] > at[n - n_new:, None]  # a query sees the rows up to its own
        for layer in range(case["layers"]):
            for head in range(case["kv_heads"]):
                keys, queries = _rope(k[b, layer, head, :n], at), _rope(q[layer, b, head].double(), at[n - n_new:])
                scores = (queries @ keys.T / math.sqrt(d)).masked_fill_(unseen, -math.inf)
                out[layer, b, head] = torch.softmax(scores, dim=-1) @ v[b, layer, head, :n]
    return out.reshape(st["q"].shape), k, v
