"""Performance cases of the library: the passes its users run, through the public Python entry points.

A case names one kind of pass and its shape:
  kind     "prefill" (forward), "train" (forward + backward on one workspace), "decode" (one cached decoding step)
  variant  "plain", "gated" (scalar gates), "normalized" (augmented ones column, final division),
           "routed" (user-supplied cells and types)
  d, batch, heads, T, d_k, d_v, chunk, dtype   as SmatPlan takes them

The listed shapes are those of the repository's own workloads (paper_2609_36062_b200/synth.py, bench.py) where it has
one.  Lengths are multiples of the chunk width only: a prompt is as long as it is, so a block boundary that is not a
whole 128-token tile is as ordinary as one that is; training sequences are cut to whole multiples of 256.
"""
import math

import torch

from paper_2609_36062_b200 import binding


def _case(name, kind, d, batch, heads, T, chunk=128, d_k=128, d_v=128, dtype="bf16", variant="plain"):
    return {"name": name, "kind": kind, "variant": variant, "d": d, "batch": batch, "heads": heads, "T": T, "d_k": d_k,
            "d_v": d_v, "chunk": chunk, "dtype": dtype}


def listed():
    return [
        # fp32 layer of one small head: a unit-sized model, a test, a debugging session; launches and latency only
        _case("f32_512_d2_train", "train", 2, 1, 1, 512, 64, 64, 64, "f32"),
        # a short-context batch: 32 heads of 4096 tokens
        _case("prefill_4k_d3", "prefill", 3, 4, 8, 4096, 64),
        # a short prompt of no particular length with the paper's normalised output (block boundary inside a tile)
        _case("prefill_5056_d3_normalized", "prefill", 3, 4, 8, 5056, 64, variant="normalized"),
        # medium context, richest mask of the default configurations
        _case("prefill_16k_d4", "prefill", 4, 2, 16, 16384),
        # the same with content-based routing handed in as arrays
        _case("prefill_16k_d4_routed", "prefill", 4, 2, 16, 16384, variant="routed"),
        # one long document: plain causal linear attention, a medium and the richest mask
        _case("prefill_64k_d1", "prefill", 1, 1, 16, 65536),
        _case("prefill_64k_d3", "prefill", 3, 1, 16, 65536),
        _case("prefill_64k_d4", "prefill", 4, 1, 16, 65536),
        # one layer's training step, forward and backward on the kept tables
        _case("train_8k_d3", "train", 3, 8, 16, 8192, 64),
        # the same for the gated variant (gradients of the gates among the outputs)
        _case("train_4k_d3_gated", "train", 3, 4, 8, 4096, 64, variant="gated"),
        # serving, one token: a few sequences (latency), and a full batch
        _case("decode_b4_2k_d3", "decode", 3, 4, 16, 2048, 64),
        _case("decode_b32_2k_d3", "decode", 3, 32, 16, 2048, 64),
    ]


MAX_STATES = 165_000          # states of all heads in both tables, the most a listed case has (prefill_64k_d4)
MAX_ROWS = 16 * 65536         # tokens of all heads


def _boundary(T, chunk):
    return chunk * (T // (2 * chunk))


def _states(d, n):
    """(P, B): profile cells and types of the default field size, the smallest prime q with q^d >= n."""
    if d == 1:
        return 1, 1
    q = 2
    while q ** d < n or any(q % f == 0 for f in range(2, int(math.isqrt(q)) + 1)):
        q += 1
    P = q ** (d - 1)
    return P, q * (P - 1) // (q - 1)


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    while True:
        kind = rng.choices(("prefill", "train", "f32", "decode"), weights=(7, 2, 1, 2))[0]
        if kind == "decode":
            c = _case("", "decode", rng.choice((1, 2, 3)), round(_log_uniform(rng, 1, 32)), rng.choice((8, 16)),
                      256 * rng.randint(4, 12), 64)
        elif kind == "f32":
            chunk, dk = rng.choice((32, 64)), rng.choice((64, 128))
            c = _case("", "train", rng.choice((1, 2, 3)), 1, rng.randint(1, 8), chunk * round(_log_uniform(rng, 256, 2048) / chunk),
                      chunk, dk, rng.choice((64, dk)), "f32")
        elif kind == "train":
            variant = rng.choice(("plain", "gated"))
            c = _case("", "train", rng.choice((2, 3, 4)), rng.randint(1, 8), rng.choice((8, 16)),
                      256 * round(_log_uniform(rng, 2048, 8192) / 256), rng.choice((64, 128)), variant=variant)
        else:
            variant, T = rng.choice(("plain", "plain", "normalized", "routed")), _log_uniform(rng, 2048, 65536)
            d = rng.choice((2, 3, 4)) if variant == "routed" else rng.choice((1, 2, 3, 4))
            chunk = rng.choice((64, 128)) if T < 16384 else 128      # long contexts are cut into the widest chunks
            c = _case("", "prefill", d, rng.randint(1, 4), rng.choice((8, 16)), chunk * round(T / chunk), chunk,
                      variant=variant)
        del c["name"]
        bh, P_B = c["batch"] * c["heads"], sum(_states(c["d"], _boundary(c["T"], c["chunk"])))
        most = 0.5 if c["kind"] == "train" else 1.0   # a training step goes over its tables twice as often
        if c["kind"] == "decode" or (bh * P_B <= most * MAX_STATES and bh * c["T"] <= MAX_ROWS):
            return c


def _flags(case):
    f = {"gated": binding.FLAG_GATED, "normalized": binding.FLAG_NORMALIZED}.get(case["variant"], 0)
    if case["kind"] == "train" and case["dtype"] == "bf16":
        f |= binding.FLAG_KEEP_FORWARD_TABLES      # the backward follows its forward on the same workspace
    return f


def prepare(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    B, H, T, dk, dv = case["batch"], case["heads"], case["T"], case["d_k"], case["d_v"]
    dtype = torch.bfloat16 if case["dtype"] == "bf16" else torch.float32

    def normal(*shape):
        return torch.randn(*shape, generator=g, device="cuda", dtype=torch.float32)

    def feature(*shape):      # rows of Q and K: unit length (non-negative features for the normalised output)
        x = normal(*shape)
        if case["variant"] == "normalized":
            return (x.abs_() / math.sqrt(shape[-1])).to(dtype)
        return torch.nn.functional.normalize(x, dim=-1).to(dtype)

    plan = binding.SmatPlan(B, H, T, dk, dv, case["d"], case["chunk"], case["dtype"], flags=_flags(case))
    st = {"case": case, "plan": plan}
    if case["kind"] == "decode":
        cache = plan.decode_cache()
        plan.decode_begin(feature(B, H, T, dk), normal(B, H, T, dv).to(dtype), cache, workspace=plan.workspace())
        geo = plan.geometry()
        tokens = 16           # rows of the tokens that are decoded one after the other
        st.update(cache=cache, first=geo.n, count=geo.m, step=0,
                  running=cache[cache.numel() - B * H * dk * dv * 4:].view(torch.float32).view(B, H, dk, dv),
                  q=[feature(B, H, dk) for _ in range(tokens)], k=[feature(B, H, dk) for _ in range(tokens)],
                  v=[normal(B, H, dv).to(dtype) for _ in range(tokens)])
        return st
    st.update(q=feature(B, H, T, dk), k=feature(B, H, T, dk), v=normal(B, H, T, dv).to(dtype),
              ws=plan.workspace(for_backward=case["kind"] == "train"))
    if case["kind"] == "train":
        st["do"] = normal(B, H, T, dv).to(dtype)
    if case["variant"] == "gated":      # gates in [0.998, 1): a memory of about a thousand tokens, so that the routed
        # long-range keys still count (with gates of 0.95 nothing reaches across the block boundary)
        st["log_a"] = torch.log(torch.rand(B * H, T, generator=g, device="cuda") * 0.002 + 0.998)
    if case["variant"] == "routed":     # every token hashed to a cell, every query to a type
        geo = plan.geometry()
        st["prof"] = torch.randint(geo.P, (B * H, geo.n), generator=g, device="cuda", dtype=torch.int32)
        st["type"] = torch.randint(geo.B, (B * H, geo.m), generator=g, device="cuda", dtype=torch.int32)
    return st


def run(st):
    plan, case = st["plan"], st["case"]
    if case["kind"] == "decode":
        i, st["step"] = st["step"], st["step"] + 1
        r = i % len(st["q"])
        o = plan.decode_step(st["q"][r], st["k"][r], st["v"][r], st["first"] + i % st["count"], st["cache"])
        return {"o": o, "state": st["running"]}
    q, k, v, ws = st["q"], st["k"], st["v"], st["ws"]
    if case["kind"] == "prefill":
        if case["variant"] == "normalized":
            return {"O": plan.forward_normalized(q, k, v, workspace=ws)}
        if case["variant"] == "routed":
            return {"O": plan.forward(q, k, v, workspace=ws, prof=st["prof"], type=st["type"])}
        return {"O": plan.forward(q, k, v, workspace=ws)}
    if case["variant"] == "gated":
        O = plan.forward_gated(q, k, v, st["log_a"], workspace=ws)
        dQ, dK, dV, dlog_a = plan.backward_gated(q, k, v, st["log_a"], st["do"], workspace=ws)
        return {"O": O, "dQ": dQ, "dK": dK, "dV": dV, "dlog_a": dlog_a}
    O = plan.forward(q, k, v, workspace=ws)
    dQ, dK, dV = plan.backward(q, k, v, st["do"], workspace=ws)
    return {"O": O, "dQ": dQ, "dK": dK, "dV": dV}


def work(case):
    """Inputs read once, outputs written once; multiply-adds of the chunkwise method in its 128-token form (two
    operations each), and the additions of the tables taken one coordinate at a time (about (d - 2) q^d a state entry)."""
    bh, T, r, p, d = case["batch"] * case["heads"], case["T"], case["d_k"], case["d_v"], case["d"]
    e, rp = 2 if case["dtype"] == "bf16" else 4, case["d_k"] * case["d_v"]
    if case["kind"] == "decode":
        # running state read and written (fp32), one type state read (bf16; fp32 for d = 1), the token's rows
        return {"bytes": bh * (2 * rp * 4 + rp * (2 if d > 1 else 4) + (2 * r + 2 * p) * e), "flops": bh * 6 * rp}
    n = _boundary(T, case["chunk"])
    q = round(_states(d, n)[0] ** (1 / (d - 1))) if d > 1 else 0
    additions = (d - 2) * q ** d * rp if d > 2 else 0
    by, fl = T * (2 * r + 2 * p) * e, T * 129 * (r + p) + 4 * T * rp + (2 * T * rp + additions if d > 1 else 0)
    if case["kind"] == "train":
        by += T * (4 * r + 3 * p) * e
        fl += T * 129 * (3 * r + 2 * p) + 6 * T * rp + (6 * T * rp + additions if d > 1 else 0)
    if case["variant"] == "gated":
        by += T * 4 * (3 if case["kind"] == "train" else 1)
    if case["variant"] == "routed":
        by += T * 4
    return {"bytes": bh * by, "flops": bh * fl}


def tolerance(case):
    """About four times what the default path differs by from the fp64 definition or, at sizes beyond that, from the
    library's own fp32-ALU form: fp32 2e-7 (another order of the sums: a few e-7 more), bf16 2.4e-3 to 3.4e-3."""
    if case["dtype"] == "f32":
        return {"rel": 1e-5}
    if case["kind"] == "train" and case["variant"] == "gated":
        return {"rel": 3e-2}      # the gate gradient: a suffix sum of differences of rounded products
    return {"rel": 1e-2}
