"""The work that a user of the library has it do, as a list of timed cases.

Three kinds, all through the public entry points:

  prefill  the causal forward over whole sequences (`lla_forward`, `lla_forward_f32`) or over a chunk of queries
           appended to existing keys (`lla_forward_ex` with `q_rows`, grouped heads, a sliding window)
  decode   one query per (sequence, head) over a key/value cache (`lla_decode`, or `lla_decode_ex` on a paged cache)
  train    the forward that saves what the backward pass needs, then the backward pass

`recipe` names the distribution of the inputs:

  iid         q, k ~ N(0, 1/d), v ~ N(0, 1): the synthetic prefill and decode workloads
  regression  keys N(0, I/d), values A_s k_j + 0.1 noise with the map A_s redrawn every 512 tokens, query i = key i + 1:
              the test-time-regression workload
  normed      q, k ~ N(0, 1) per entry, as behind a query/key normalisation: scores of unit variance, so weights that are
              far from uniform
"""
import math

import torch

import paper_2510_01450_b200 as L

SEGMENT = 512


def _case(name, kind, B, H, n, d, **kw):
    c = {"name": name, "kind": kind, "dtype": "bf16", "recipe": "iid", "B": B, "H": H, "kv_heads": H, "n": n, "d": d,
         "q_rows": n if kind != "decode" else 1, "window": 0, "page": 0, "len_min": n, "lam": 1e-3}
    c.update(kw)
    return c


def listed():
    return [
        # the smallest call: one fp32 head; launches and the longest chain of dependent steps are all of it
        _case("prefill_f32_n256_d16", "prefill", 1, 1, 256, 16, dtype="f32", lam=1e-2),
        # fp32 inputs at an ordinary head size, a length that is no multiple of any tile
        _case("prefill_f32_n1000_d64", "prefill", 2, 4, 1000, 64, dtype="f32"),
        # short prompts in a batch: few key blocks a row, and a tenth of the rows are solved directly
        _case("prefill_n1024_d64", "prefill", 4, 8, 1024, 64),
        # the test-time-regression shape
        _case("prefill_n4096_d64", "prefill", 2, 16, 4096, 64, recipe="regression", lam=1e-2),
        # long context
        _case("prefill_n16384_d128", "prefill", 1, 16, 16384, 128),
        # serving: the next chunk of a long prompt against the keys already there, grouped heads, ragged sizes
        _case("chunk_n5003_q257_d128_gqa", "prefill", 2, 16, 5003, 128, kv_heads=4, q_rows=257, recipe="normed"),
        # one sequence being generated: latency
        _case("decode_b1_d64", "decode", 1, 16, 4096, 64, len_min=3001),
        # a full batch being generated
        _case("decode_b64_d64", "decode", 64, 16, 8192, 64, len_min=1024),
        # serving with a paged cache and grouped heads at the larger head size
        _case("decode_b24_d128_paged_gqa", "decode", 24, 16, 5000, 128, kv_heads=4, len_min=300, page=256, recipe="normed"),
        # training steps: short ragged sequences, the regression shape, long context at the larger head size
        _case("train_n1000_d64", "train", 4, 8, 1000, 64),
        _case("train_n4096_d64", "train", 2, 16, 4096, 64, recipe="regression", lam=1e-2),
        _case("train_n16384_d128", "train", 1, 16, 16384, 128),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """A case from the same ranges: sizes spread over their logarithm, odd ones among them."""
    most = 16 * 16384 * 16384 * 128      # heads x rows x keys x head size of the largest listed case
    while True:
        kind = rng.choice(["prefill", "prefill", "f32", "chunk", "decode", "decode", "train", "train"])
        if kind == "f32":
            d = rng.choice([16, 64, 128])
            c = _case("", "prefill", rng.randint(1, 2), rng.choice([1, 2, 4, 8]), _log_int(rng, 100, 2000), d, dtype="f32",
                      lam=rng.choice([1e-3, 1e-2]))
        elif kind == "decode":
            H = rng.choice([8, 16, 32])
            page = rng.choice([0, 0, 128, 256])
            n = _log_int(rng, 512, 8192)
            c = _case("", "decode", _log_int(rng, 1, 64), H, n, rng.choice([64, 128]), page=page,
                      kv_heads=H // rng.choice([1, 1, 4]), len_min=rng.randint(max(256, n // 8), n),
                      recipe=rng.choice(["iid", "normed"]), lam=rng.choice([1e-3, 1e-2]))
        elif kind == "chunk":
            H = rng.choice([8, 16])
            n = _log_int(rng, 3000, 16384)
            c = _case("", "prefill", rng.randint(1, 4), H, n, rng.choice([64, 128]), q_rows=_log_int(rng, 16, 1024),
                      kv_heads=H // rng.choice([1, 2, 4]), window=rng.choice([0, 0, rng.randint(1024, n)]),
                      recipe=rng.choice(["iid", "normed"]), lam=rng.choice([1e-3, 1e-2]))
        else:
            c = _case("", kind, rng.randint(1, 4), rng.choice([4, 8, 16]), _log_int(rng, 128, 16384), rng.choice([64, 128]),
                      recipe=rng.choice(["iid", "regression"]), lam=rng.choice([1e-3, 1e-2]))
        del c["name"]
        if c["B"] * c["H"] * c["q_rows"] * c["n"] * c["d"] <= most:
            return c


def _lens(c):
    """Cache lengths, evenly spread over the case's range (their order is the seed's)."""
    B, lo, hi = c["B"], c["len_min"], c["n"]
    return [hi if B == 1 and lo == hi else (lo + hi) // 2 if B == 1 else lo + (hi - lo) * b // (B - 1) for b in range(B)]


def _prefill_inputs(c, gen):
    B, H, Hk, n, d, nq = c["B"], c["H"], c["kv_heads"], c["n"], c["d"], c["q_rows"]
    dt = torch.float32 if c["dtype"] == "f32" else torch.bfloat16

    def randn(*shape):
        return torch.randn(shape, generator=gen, device="cuda", dtype=torch.float32)

    if c["recipe"] == "regression":
        keys = randn(B, H, n + 1, d) / math.sqrt(d)
        k, q = keys[:, :, :n], keys[:, :, 1:]
        v = 0.1 * randn(B, H, n, d)
        for s in range(0, n, SEGMENT):
            a = randn(B, H, d, d) / math.sqrt(d)
            v[:, :, s:s + SEGMENT] += k[:, :, s:s + SEGMENT] @ a.transpose(-1, -2)
    else:
        sd = 1.0 if c["recipe"] == "normed" else 1.0 / math.sqrt(d)
        q, k, v = randn(B, H, nq, d) * sd, randn(B, Hk, n, d) * sd, randn(B, Hk, n, d)
        if d == 16:
            v = v / math.sqrt(d)
    return [t.to(dt).contiguous() for t in (q, k, v)]


def prepare(case, seed):
    """Inputs, output buffers and the scratch that a program keeps between calls."""
    c = case
    gen = torch.Generator(device="cuda").manual_seed(seed)
    B, H, Hk, n, d = c["B"], c["H"], c["kv_heads"], c["n"], c["d"]
    s = {"c": c, "scale": 1.0 / math.sqrt(d)}

    def empty(*shape, dtype=torch.float32):
        return torch.empty(shape, dtype=dtype, device="cuda")

    def scratch(nbytes):
        return torch.empty(nbytes, dtype=torch.uint8, device="cuda") if nbytes else None

    if c["kind"] == "decode":
        lens = torch.tensor(_lens(c), dtype=torch.int32, device="cuda")
        lens = lens[torch.randperm(B, generator=gen, device="cuda")]
        sd = 1.0 if c["recipe"] == "normed" else 1.0 / math.sqrt(d)
        if c["page"]:
            per = (n + c["page"] - 1) // c["page"]
            rows = (B * per, Hk, c["page"], d)
            s["table"] = torch.randperm(B * per, generator=gen, device="cuda").to(torch.int32).reshape(B, per)
        else:
            rows = (B, Hk, n, d)
        s["k"] = (torch.randn(rows, generator=gen, device="cuda") * sd).to(torch.bfloat16)
        s["v"] = torch.randn(rows, generator=gen, device="cuda").to(torch.bfloat16)
        s["q"] = (torch.randn((B, H, d), generator=gen, device="cuda") * sd).to(torch.bfloat16)
        s["lens"], s["out"] = lens, empty(B, H, d, dtype=torch.bfloat16)
        s["ws_bytes"] = L.lla_decode_workspace_bytes(B, H, n, d, d, L.LLA_BF16, L.lla_decode_default_splits(B, H, n))
        s["ws"] = scratch(s["ws_bytes"])
        return s

    s["q"], s["k"], s["v"] = _prefill_inputs(c, gen)
    nq = c["q_rows"]
    s["ws_bytes"] = L.lla_forward_workspace_bytes(B, H, n, d, d, L.LLA_F32 if c["dtype"] == "f32" else L.LLA_BF16)
    s["ws"] = scratch(s["ws_bytes"])
    train = c["kind"] == "train"
    s["out"] = empty(B, H, nq, d, dtype=torch.float32 if train or c["dtype"] == "f32" else torch.bfloat16)
    if train:
        s["dout"] = torch.randn((B, H, n, d), generator=gen, device="cuda")
        s["rho"], s["stats"] = empty(B, H, n, d), empty(B, H, n, 3)
        s["dq"], s["dk"], s["dv"] = empty(B, H, n, d), empty(B, H, n, d), empty(B, H, n, d)
        s["bws_bytes"] = L.lla_backward_workspace_bytes(B, H, n, d)
        s["bws"] = scratch(s["bws_bytes"])
    return s


def run(s):
    c = s["c"]
    B, H, Hk, n, d = c["B"], c["H"], c["kv_heads"], c["n"], c["d"]
    scale, lam = s["scale"], c["lam"]
    stream = torch.cuda.current_stream().cuda_stream
    if c["kind"] == "decode":
        if c["page"] or Hk != H or d != 64:
            # a serving loop: its own scratch, its own page table
            paged = {"block_table": s["table"], "page_size": c["page"], "max_pages": s["table"].shape[1],
                     "num_pages": s["k"].shape[0]} if c["page"] else {}
            L.lla_decode_ex(s["q"], s["k"], s["v"], s["lens"], s["out"], B, H, n, d, d, scale, lam, kv_heads=Hk,
                            workspace=s["ws"], workspace_bytes=s["ws_bytes"], stream=stream, **paged)
        else:
            L.lla_decode(s["q"], s["k"], s["v"], s["lens"], s["out"], B, H, n, d, d, scale, lam, stream=stream)
        return s["out"]
    if c["kind"] == "train":
        L.lla_forward_ex(s["q"], s["k"], s["v"], s["out"], B, H, n, d, d, scale, lam, out_dtype=L.LLA_F32, rho=s["rho"],
                         stats=s["stats"], workspace=s["ws"], workspace_bytes=s["ws_bytes"], stream=stream)
        L.lla_backward_ex(s["q"], s["k"], s["v"], s["out"], s["dout"], s["rho"], s["stats"], s["dq"], s["dk"], s["dv"],
                          B, H, n, d, scale, lam, workspace=s["bws"], workspace_bytes=s["bws_bytes"], stream=stream)
        return {"out": s["out"], "dq": s["dq"], "dk": s["dk"], "dv": s["dv"]}
    if c["dtype"] == "f32":
        L.lla_forward_f32(s["q"], s["k"], s["v"], s["out"], B, H, n, d, d, scale, lam, stream=stream)
    elif c["q_rows"] != n or Hk != H or c["window"]:
        L.lla_forward_ex(s["q"], s["k"], s["v"], s["out"], B, H, n, d, d, scale, lam, q_rows=c["q_rows"], kv_heads=Hk,
                         window=c["window"], workspace=s["ws"], workspace_bytes=s["ws_bytes"], stream=stream)
    else:
        L.lla_forward(s["q"], s["k"], s["v"], s["out"], B, H, n, d, d, scale, lam, stream=stream)
    return s["out"]


def work(case):
    """Bytes: every input read once, every output written once.  Flops per visible (query, key) pair of a prefill: the
    score 2d, the key mean 2d, one application of the row's operator 4d, the coefficient 2d, the output 2d = 12d; of a
    backward pass: score, value product, key mean and right-hand side 8d, one application of the operator 4d, the two
    key products 4d, dq 2d, dk 6d, dv 2d = 26d; per (query, key) of a decode step: the symmetric moment d^2, the
    value moment 2 d^2, score and first moments 6d."""
    c = case
    B, H, Hk, n, d, nq = c["B"], c["H"], c["kv_heads"], c["n"], c["d"], c["q_rows"]
    size = 4 if c["dtype"] == "f32" else 2
    if c["kind"] == "decode":
        keys = sum(_lens(c))
        return {"bytes": keys * Hk * 2 * d * size + 2 * B * H * d * size, "flops": keys * H * (3 * d * d + 6 * d)}
    w = c["window"] or n
    first = n - nq
    pairs = B * H * sum(min(i + 1, w) for i in range(first, n))
    seen = min(n, w + nq)
    fwd = (2 * B * H * nq * d + 2 * B * Hk * seen * d) * size
    if c["kind"] == "train":
        # q, k, v in; out, rho, stats written by the forward and read by the backward; dout in; three gradients out
        per = B * H * n
        return {"bytes": per * (3 * d * size + 3 * d * 4 + 4 * (3 * d + d + 3)), "flops": pairs * 38 * d}
    return {"bytes": fwd, "flops": pairs * 12 * d}


def tolerance(case):
    """About four times what the outputs of the listed and of drawn cases differ from the same formulas in float64 (rel:
    2-norm; max: largest difference over the root mean square).  Gradients and fp32 outputs of bf16 inputs: up to 1.5e-4
    and 1.9e-3 (the solver stops at a relative residual of 1e-4); fp32 inputs: up to 4.5e-7 and 9e-6; bf16 outputs
    against the float64 result rounded to bf16: up to 1.0e-3 and 7.8e-3 (a last place where the rounding falls the
    other way)."""
    if case["kind"] == "train":
        return {"rel": 6e-4, "max": 8e-3}
    if case["dtype"] == "f32":
        return {"rel": 2e-6, "max": 4e-5}
    return {"rel": 4e-3, "max": 3.1e-2}
