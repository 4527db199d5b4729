"""The work that users of this library have it do, as cases that can be timed and compared.

A case names one call of a public entry point with its sizes, its tensor type and its options; prepare() makes what a
user's program holds before the call, run() makes the call.  Values are drawn as synth.py draws them, on the device.
"""
from __future__ import annotations

import math

import torch

from paper_2509_23436_b200 import binding

_DTYPES = {"bf16": torch.bfloat16, "f32": torch.float32}
_CODES = {"bf16": binding.LOT_BF16, "f32": binding.LOT_F32}


def _case(name, op, dtype, B, H, n, d, r, eps, iters, **options):
    """op: fwd (lot_attention_fwd_ex), plain (lot_attention_fwd), bwd (lot_attention_bwd), var (lot_attention_fwd_var).

    nk: keys per slice (var only; n otherwise).  mask: seeded key lengths in [n/2, n].  mixture: queries and keys from
    four clusters (peaked similarities).  cls: the class-token row.  weights: token weights on both sides.  warm: the
    iteration starts from the potentials of an earlier call and gives its own back.
    """
    c = dict(op=op, dtype=dtype, B=B, H=H, n=n, nk=n, d=d, r=r, eps=eps, iters=iters,
             mask=False, mixture=False, cls=False, weights=False, warm=False)
    c.update(options)
    if name is not None:
        c["name"] = name
    return c


def listed():
    return [
        # one tiny head in float32 through the plain signature: a call that is all launch and latency
        _case("tiny-f32", "plain", "f32", 1, 1, 64, 16, 8, 0.1, 50),
        # image classification, a batch of 32 through one DeiT-Tiny-shaped layer: inference in bf16 ...
        _case("image-bf16", "fwd", "bf16", 32, 3, 197, 64, 16, 0.1, 10),
        # ... the same layer with its class token kept as a softmax row ...
        _case("image-cls-bf16", "var", "bf16", 32, 3, 197, 64, 16, 0.1, 10, cls=True),
        # ... and its training step's backward
        _case("image-bwd-bf16", "bwd", "bf16", 32, 3, 197, 64, 16, 0.1, 10),
        # text, a padded batch through one BERT-base-shaped layer, in both tensor types
        _case("text-bf16", "fwd", "bf16", 16, 12, 512, 64, 32, 0.05, 20, mask=True),
        _case("text-f32", "fwd", "f32", 16, 12, 512, 64, 32, 0.05, 20, mask=True),
        # cross-attention of a short query set to a longer weighted key set, warm-started, in float32
        _case("cross-f32", "var", "f32", 8, 8, 333, 64, 32, 0.1, 5, nk=1531, weights=True, warm=True),
        # long context, the headline sweep's three lengths
        _case("long4k-bf16", "fwd", "bf16", 1, 16, 4096, 64, 64, 0.1, 10),
        _case("long16k-bf16", "fwd", "bf16", 1, 16, 16384, 64, 64, 0.1, 10),
        _case("long64k-bf16", "fwd", "bf16", 1, 16, 65536, 64, 64, 0.1, 10),
        # long-context training: the backward of the shortest of them
        _case("long4k-bwd-bf16", "bwd", "bf16", 1, 16, 4096, 64, 64, 0.1, 10),
        # wide heads, high rank and peaked similarities: the rank and iteration stress of the configurations
        _case("stress-bf16", "fwd", "bf16", 4, 8, 16384, 128, 256, 0.1, 20, mixture=True),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _load(c):
    """A measure of a case's cost: matrix entries touched over all iterations and products."""
    per = c["r"] * (c["iters"] + 3 + c["d"] / 32.0)
    return c["B"] * c["H"] * (c["n"] + c["nk"]) * per * (3 if c["op"] == "bwd" else 1) * (2 if c["dtype"] == "f32" else 1)


def draw(rng):
    """One more case: batch and heads, sequence length (log-uniform, odd ones too), rank, width, iterations, options."""
    most = 0.5 * _load(next(c for c in listed() if c["name"] == "stress-bf16"))
    while True:
        op = rng.choice(["fwd", "fwd", "fwd", "bwd", "var"])
        dtype = rng.choice(["bf16", "bf16", "f32"])
        n = _log_int(rng, 64, 65536 if op == "fwd" else 16384)
        if rng.random() < 0.4:
            n = max(64, n // 64 * 64)
        B, H = _log_int(rng, 1, 32), rng.choice([3, 6, 8, 12, 16])
        d = rng.choice([32, 64, 64, 64, 128])
        r = rng.choice([8, 16, 16, 32, 32, 64, 64, 128, 256, rng.randint(9, 100)])
        eps = rng.choice([0.05, 0.1, 0.1]) if op == "bwd" or dtype == "f32" else rng.choice([0.02, 0.05, 0.1, 0.1])
        c = _case(None, op, dtype, B, H, n, d, r, eps, rng.choice([5, 10, 10, 20, 20, 50]), mixture=rng.random() < 0.25)
        if op == "var":
            kind = rng.choice(["cls", "cross", "cross"])
            if kind == "cls":
                c["cls"] = True
            else:
                c["nk"] = _log_int(rng, 64, 16384)
                c["weights"], c["warm"] = rng.random() < 0.5, rng.random() < 0.5
        else:
            c["mask"] = rng.random() < 0.4
        tokens = B * H * (c["n"] + c["nk"])
        if tokens * d <= (1 << 29) and _load(c) <= most:
            return c


def prepare(case, seed):
    c, dev = case, torch.device("cuda")
    gen = torch.Generator(device=dev)
    gen.manual_seed(int(seed))
    dt, code = _DTYPES[c["dtype"]], _CODES[c["dtype"]]
    B, H, n, nk, d, r = c["B"], c["H"], c["n"], c["nk"], c["d"], c["r"]
    std = d ** -0.5

    def normal(*shape):
        return torch.randn(*shape, generator=gen, device=dev, dtype=torch.float32)

    if c["mixture"]:
        means = normal(B, H, 4, d) * (2.0 * std)

        def tokens(m):
            which = torch.randint(0, 4, (B, H, m, 1), generator=gen, device=dev)
            return (torch.gather(means, 2, which.expand(B, H, m, d)) + normal(B, H, m, d) * (0.5 * std)).to(dt)
    else:
        def tokens(m):
            return (normal(B, H, m, d) * std).to(dt)

    s = dict(op=c["op"], eps=c["eps"], iters=c["iters"], cls=c["cls"], key_len=None)
    s["q"], s["k"] = tokens(n), tokens(nk)
    s["v"] = (normal(B, H, nk, d) * std).to(dt)
    # the tiny configuration scales its pivots like its tokens, the others draw them N(0,1)
    s["z"] = normal(H, r, d) * (std if c["op"] == "plain" else 1.0)
    s["beta"] = torch.softmax(normal(H, r), dim=-1)
    if c["mask"]:
        s["key_len"] = torch.randint(nk // 2, nk + 1, (B,), generator=gen, device=dev, dtype=torch.int32)
    if c["op"] == "bwd":
        s["dout"] = normal(B, H, n, d).to(dt)
        need = binding.lot_bwd_workspace_bytes(B, H, n, d, r, code, c["iters"])
    elif c["op"] == "var":
        s["a"] = s["b"] = s["g1_in"] = s["g2_in"] = s["g1"] = s["g2"] = None
        if c["weights"]:
            s["a"] = torch.softmax(0.5 * normal(B, H, n), dim=-1)
            s["b"] = torch.softmax(0.5 * normal(B, H, nk), dim=-1)
        if c["warm"]:
            s["g1_in"], s["g2_in"] = c["eps"] * normal(B, H, r), c["eps"] * normal(B, H, r)
            s["g1"] = torch.empty(B, H, r, device=dev, dtype=torch.float32)
            s["g2"] = torch.empty(B, H, r, device=dev, dtype=torch.float32)
        need = binding.lot_var_workspace_bytes(B, H, n, nk, d, r, code)
    else:
        need = binding.lot_workspace_bytes(B, H, n, d, r, code)
    if c["op"] != "bwd":
        s["out"] = torch.empty_like(s["q"])
    if c["op"] != "plain":
        s["ws"] = torch.empty(max(need, 256), device=dev, dtype=torch.uint8)
    return s


def run(s):
    args = (s["q"], s["k"], s["v"], s["z"], s["beta"])
    if s["op"] == "plain":
        return binding.lot_attention_fwd(*args, s["eps"], s["iters"], out=s["out"])
    if s["op"] == "fwd":
        return binding.lot_attention_fwd_ex(*args, s["key_len"], s["eps"], s["iters"], out=s["out"], ws=s["ws"])[0]
    if s["op"] == "bwd":
        return binding.lot_attention_bwd(*args, s["key_len"], s["dout"], s["eps"], s["iters"], ws=s["ws"])[:5]
    binding.lot_attention_fwd_var(*args, s["eps"], s["iters"], a=s["a"], b=s["b"], key_len=s["key_len"],
                                  g1_in=s["g1_in"], g2_in=s["g2_in"], cls=s["cls"], cls_tau=1.0, out=s["out"],
                                  g1_out=s["g1"], g2_out=s["g2"], ws=s["ws"])
    return [t for t in (s["out"], s["g1"], s["g2"]) if t is not None]


def work(case):
    c = case
    slices, both = c["B"] * c["H"], c["n"] + c["nk"]
    size = 2 if c["dtype"] == "bf16" else 4
    small = c["H"] * c["r"] * (c["d"] + 1) * 4 * (2 if c["op"] == "bwd" else 1)
    if c["mask"]:
        small += 4 * c["B"]
    if c["weights"]:
        small += 4 * slices * both
    if c["warm"]:
        small += 16 * slices * c["r"]
    # q and out, k and v; the backward also reads the output's gradient and writes dq, dk, dv in place of out
    rows = 2 * both if c["op"] != "bwd" else 3 * c["n"] + 4 * c["nk"]
    # similarities and the two apply products; the backward repeats three of them and has eight products of its own
    products = 2 * both * c["r"] * c["d"] * (2 if c["op"] != "bwd" else 5.5)
    # a multiply-add for the row sum and one for the column sum of each entry and iteration, twice that in reverse
    passes = 4 * both * c["r"] * (c["iters"] + 1) * (1 if c["op"] != "bwd" else 3)
    return {"bytes": slices * rows * c["d"] * size + small, "flops": slices * (products + passes)}


def tolerance(case):
    """bf16 tensors: the rounding of the tensors; float32 tensors: float32 sums, twice that through the reverse sweep."""
    if case["dtype"] == "bf16":
        return {"rel": 1e-2, "max": 0.1}
    return {"rel": 2e-5 if case["op"] == "bwd" else 1e-5, "max": 5e-4}
