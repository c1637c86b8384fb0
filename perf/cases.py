"""The work that a user of this library has it do, as cases that can be timed and compared.

Two operations of one layer: the prefill (`ha_la_prefill`: all tokens of the prompts, state handed in and out) and the
decoding step (`ha_la_decode`: one token per sequence on the state the prefill left, in place).  Both are called the
way a serving program calls them: tensors in hand, the scratch workspace and the status word kept from call to call,
outputs allocated by the call.  Values follow the recipe of paper_2609_32114_b200/synth.py: unit-norm q and k,
v ~ N(0, 1), beta = sigmoid(N(0, 1)), log-gate = -softplus(N(0, 1) + gate_shift), states ~ N(0, std 0.02) (prefill) or
std 0.5 (decode), q / k / v in bf16 or fp32, everything else fp32.
"""
import math
import random

import torch

import paper_2609_32114_b200 as ha


def _prefill(name, variant, hk, hv, d=128, dtype="bf16", rows=1, tokens=0, packed=0, lo=0, hi=0, len_seed=0,
             h0=False, gate_shift=2.0):
    """`rows` prompts of `tokens` tokens each, or, with `packed` > 0, that many prompts of lo..hi tokens end to end."""
    c = dict(op="prefill", variant=variant, dtype=dtype, d=d, hk=hk, hv=hv, rows=rows, tokens=tokens, packed=packed,
             lo=lo, hi=hi, len_seed=len_seed, h0=h0, gate_shift=gate_shift)
    return dict(c, name=name) if name else c


def _decode(name, variant, n, hk, hv, d=128, dtype="bf16"):
    """One new token for each of n running sequences."""
    c = dict(op="decode", variant=variant, dtype=dtype, d=d, hk=hk, hv=hv, n=n, gate_shift=2.0)
    return dict(c, name=name) if name else c


def listed():
    return [
        # interactive decoding of a single sequence: the smallest call there is, repeated for every token
        _decode("decode_gdn_n1", "gdn", 1, 16, 16),
        # the decoding step of a full batch (256 sequences x 16 heads: 268 MB of states)
        _decode("decode_gdn_n256", "gdn", 256, 16, 16),
        # an odd number of running sequences, per-channel gates
        _decode("decode_kda_n37", "kda", 37, 32, 32),
        # one fp32 head, d = 64: the layer as it is checked against a float64 reference
        _prefill("gdn_fp32_t256", "gdn", 1, 1, d=64, dtype="fp32", tokens=256, gate_shift=0.0),
        # a layer with small heads (d = 64), a prompt of a ragged length
        _prefill("gdn_d64_t1000", "gdn", 8, 8, d=64, tokens=1000, h0=True),
        # a short prompt: six chunks, the last one ragged
        _prefill("gdn_short_t333", "gdn", 16, 16, tokens=333),
        # the layer of a ~2B hybrid model on a 4k prompt
        _prefill("gdn_layer_t4096", "gdn", 16, 16, tokens=4096),
        # grouped values (two V-heads per q/k head), a long prompt continued from a state
        _prefill("gdn_gva_t16384", "gdn", 16, 32, tokens=16384, h0=True),
        # the KDA layer on an 8k prompt
        _prefill("kda_t8192", "kda", 32, 32, tokens=8192),
        # one tensor-parallel shard of a layer (two heads) on a long prompt
        _prefill("gdn_shard_t16384", "gdn", 2, 2, tokens=16384),
        # a batch of short KDA prompts of mixed lengths, packed
        _prefill("kda_packed_24", "kda", 16, 16, packed=24, lo=20, hi=1500, len_seed=7),
        # a packed batch of prompts from 512 to 32768 tokens, each with its own state: the largest call
        _prefill("gdn_packed_8", "gdn", 16, 16, packed=8, lo=512, hi=32768, len_seed=33, h0=True),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    variant = rng.choice(["gdn", "gdn", "kda"])
    shift = rng.choice([2.0, 2.0, 0.0, -2.0])
    kind = rng.random()
    if kind < 0.3:                                           # decoding: 1 to 300 sequences
        hk = rng.choice([2, 4, 8, 16, 32])
        hv = hk * rng.choice([1, 1, 2])
        n = _log_int(rng, 1, 300 * 16 // max(16, hv))
        return _decode(None, variant, n, hk, hv, d=rng.choice([128, 128, 64]), dtype=rng.choice(["bf16", "bf16", "fp32"]))
    if kind < 0.5:                                           # fp32 inputs or small heads: short and medium prompts
        dtype, d = rng.choice([("fp32", 64), ("fp32", 128), ("bf16", 64)])
        hk = rng.choice([1, 2, 4, 8])
        hv = hk * rng.choice([1, 1, 2])
        top = 1024 if d == 64 else 400
        if rng.random() < 0.3:
            return _prefill(None, variant, hk, hv, d=d, dtype=dtype, packed=rng.randint(2, 8), lo=8, hi=top // 2,
                            len_seed=rng.randrange(1 << 20), h0=rng.random() < 0.5, gate_shift=shift)
        return _prefill(None, variant, hk, hv, d=d, dtype=dtype, rows=rng.choice([1, 1, 2]), tokens=_log_int(rng, 16, top),
                        h0=rng.random() < 0.5, gate_shift=shift)
    most = (1 << 20) if variant == "gdn" else (1 << 19)      # tokens x V-heads of one call
    hk = rng.choice([2, 4, 8, 16, 32])
    hv = hk * rng.choice([1, 1, 1, 2]) if hk < 32 else hk
    h0 = rng.random() < 0.5
    if rng.random() < 0.4:                                   # packed prompts of mixed lengths
        n = _log_int(rng, 2, 48)
        hi = max(64, min(32768, most // (hv * n)))
        lo = _log_int(rng, 8, max(9, hi // 4))
        return _prefill(None, variant, hk, hv, packed=n, lo=lo, hi=hi, len_seed=rng.randrange(1 << 20), h0=h0,
                        gate_shift=shift)
    rows = rng.choice([1, 1, 1, 2, 4, 8])
    return _prefill(None, variant, hk, hv, rows=rows, tokens=_log_int(rng, 16, min(32768, most // (hv * rows))), h0=h0,
                    gate_shift=shift)


def _lengths(c):
    if c["packed"]:
        r = random.Random(c["len_seed"])
        return [r.randint(c["lo"], c["hi"]) for _ in range(c["packed"])]
    return [c["tokens"]] * c["rows"]


def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    c, d, hk, hv = case, case["d"], case["hk"], case["hv"]
    dt = torch.bfloat16 if c["dtype"] == "bf16" else torch.float32

    def normal(*shape):
        return torch.randn(shape, generator=gen, device="cuda", dtype=torch.float32)

    def unit(*shape):
        return torch.nn.functional.normalize(normal(*shape), dim=-1).to(dt).contiguous()

    if c["op"] == "decode":
        lead = (c["n"],)
    elif c["packed"]:
        lens = _lengths(c)
        lead = (1, sum(lens))
    else:
        lens = _lengths(c)
        lead = (c["rows"], c["tokens"])
    s = dict(q=unit(*lead, hk, d), k=unit(*lead, hk, d), v=normal(*lead, hv, d).to(dt),
             beta=torch.sigmoid(normal(*lead, hv)),
             g=-torch.nn.functional.softplus(normal(*lead, hv, *([d] if c["variant"] == "kda" else [])) + c["gate_shift"]),
             op=c["op"], variant=c["variant"])
    if c["op"] == "decode":
        s["state"] = 0.5 * normal(c["n"], hv, d, d)
        return s
    s["h0"] = 0.02 * normal(len(lens), hv, d, d) if c["h0"] else None
    s["cu_seqlens"], s["max_seqlen"] = None, 0
    if c["packed"]:
        s["cu_seqlens"] = torch.tensor([sum(lens[:i]) for i in range(len(lens) + 1)], dtype=torch.int32, device="cuda")
        s["max_seqlen"] = max(lens)
    _, keep = ha.prepare_args(s["q"], s["k"], s["v"], s["g"], s["beta"], variant=s["variant"], h0=s["h0"],
                              cu_seqlens=s["cu_seqlens"], max_seqlen=s["max_seqlen"])
    s["workspace"], s["status_word"] = keep["workspace"], keep["status_word"]
    return s


def run(s):
    if s["op"] == "decode":
        return ha.ha_la_decode(s["q"], s["k"], s["v"], s["g"], s["beta"], s["state"], variant=s["variant"])
    o, hT, _, _ = ha.ha_la_prefill(s["q"], s["k"], s["v"], s["g"], s["beta"], variant=s["variant"], h0=s["h0"],
                                   cu_seqlens=s["cu_seqlens"], max_seqlen=s["max_seqlen"], workspace=s["workspace"],
                                   status_word=s["status_word"])
    return o, hT


def work(case):
    """Each input read once, each output written once; multiply-adds counted as two operations."""
    c, d, hk, hv = case, case["d"], case["hk"], case["hv"]
    e = 2 if c["dtype"] == "bf16" else 4
    n = c["n"] if c["op"] == "decode" else len(_lengths(c))
    tokens = n if c["op"] == "decode" else sum(_lengths(c))
    state = n * hv * d * d * 4
    per_token = 2 * hk * d * e + 2 * hv * d * e + 4 * hv + 4 * hv * (d if c["variant"] == "kda" else 1)
    if c["op"] == "decode":
        return {"bytes": tokens * per_token + 2 * state, "flops": n * hv * 6.0 * d * d}
    # chunks of 64: 5 C^2 d + 3 C d^2 + C^3 / 2 multiply-adds per chunk and head (K K^T and Q K^T per q/k head)
    per_v, per_qk = 2.0 * (3 * 64 * d + 3 * d * d + 64 * 32), 2.0 * (2 * 64 * d)
    return {"bytes": tokens * per_token + (2 if c["h0"] else 1) * state, "flops": tokens * (hv * per_v + hk * per_qk)}


def tolerance(case):
    if case["dtype"] == "fp32":
        return {"rel": 1e-5}                                 # sums of fp32 products in another order
    return {"rel": 1e-2, "max": 0.15}                        # bf16 operands and outputs
