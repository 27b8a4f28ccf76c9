"""The work that programs have this library do, as measurable cases.

Three kinds, each through the public calls of `binding.SplaCache`:

  decode   one step of a generation loop: append one token per sequence and attend with its queries (`append_decode`)
  append   tokens whose outputs nobody needs go into the cache: a prompt, or a turn of a conversation (`append_tokens`)
  prefill  a chunk of tokens goes in and every position's output comes back (`prefill`)

Inputs are the ones of `synth` (needle blocks, outlier key channels, queries around one direction per KV head, ragged
lengths), drawn from the case's seed.  A state is used like a serving slot: passes continue the sequences until `room`
passes have been made; then the slot is rewound to the context it was prepared with, and the sequences grow again.
"""
from __future__ import annotations

import math

import torch

from paper_2601_22379_b200 import binding, runner, synth

DEV = "cuda:0"
DECODE_ROOM = 256        # steps a slot decodes before it is rewound

BASE = dict(kind="decode", batch=1, hq=32, hkv=8, d=128, block=64, top_k=32, context=0, context_min=0, new=1, new_min=0,
            dtype="bf16", stats16=False, window=0, stride=0, needles=0, outliers=0, drift=0.0)


def _case(name=None, **kw):
    c = dict(BASE, **kw)
    if name is not None:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest call: one sequence, one head, fp32, a few thousand tokens; latency and launches are all there is
        _case("decode 4k x1 f32", hq=1, hkv=1, d=64, top_k=8, context=4096, dtype="f32", needles=2),
        # a small serving batch at an ordinary context
        _case("decode 32k x8", batch=8, top_k=16, context=32768, needles=8, outliers=4),
        # long documents: the workload that the benchmark is quoted on
        _case("decode 128k x4", batch=4, context=131072, needles=8, outliers=4),
        # one very long document, large blocks
        _case("decode 1m x1", block=128, context=1048576, needles=16, drift=0.05),
        # a full serving batch of sequences of very different lengths
        _case("decode 64k ragged x64", batch=64, top_k=16, context=65536, context_min=4096, outliers=4),
        # the group size of the paper's own model, with the block summaries kept in 16 bits
        _case("decode 128k x4 g5 stats16", batch=4, hq=40, context=131072, needles=8, outliers=4, stats16=True),
        # the paper's strided selection windows, an odd batch and length
        _case("decode 24k x3 windows", batch=3, top_k=16, context=24601, needles=8, outliers=4, window=32, stride=16),
        # long prompts read into empty caches
        _case("append 128k x4", kind="append", batch=4, new=131072, outliers=4),
        # a turn of a conversation, of another length in each sequence, on top of the history
        _case("append turn x16", kind="append", batch=16, top_k=16, context=12288, context_min=3000, new=700, new_min=50, outliers=4),
        # a prompt from its first token on, outputs of all positions
        _case("prefill 8k", kind="prefill", new=8192, outliers=4),
        # chunked prefill of a serving loop: a chunk on top of a long context
        _case("prefill 512 on 32k x2", kind="prefill", batch=2, top_k=16, context=32768, new=512, needles=8, outliers=4),
        # a short question on a short context, small heads
        _case("prefill 77 on 500", kind="prefill", hq=16, hkv=4, d=64, block=32, top_k=8, context=500, new=77),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["decode", "decode", "append", "prefill"])
    small = rng.random() < 0.15
    hkv = rng.choice([1, 2, 4]) if small else rng.choice([2, 4, 8])
    group = rng.choice([1, 2, 4, 4, 5, 8, 8, 16])
    c = dict(kind=kind, hkv=hkv, hq=hkv * group, d=64 if small else 128, block=rng.choice([32, 64, 64, 128]),
             top_k=rng.choice([8, 16, 16, 32, 32, 64]), outliers=rng.choice([0, 4]), stats16=rng.random() < 0.25,
             dtype="f32" if small and rng.random() < 0.5 else "bf16")
    if kind == "decode":
        c["context"] = _log(rng, 1000, 1000000)
        tokens = 1000000 // hkv * 8                      # at most half of the tokens that the largest listed batch holds
        c["batch"] = max(1, min(64, _log(rng, 1, 64), tokens // c["context"]))
        if c["batch"] > 4 and rng.random() < 0.5:
            c["context_min"] = c["context"] // 8
        elif c["context"] > 80 * c["block"]:
            c["needles"] = 8
        if c["block"] >= 64 and rng.random() < 0.2:
            c["window"], c["stride"] = 32, 16
        if c["context"] > 300000:
            c["block"] = max(c["block"], 64)             # (a cache holds at most 32768 blocks per sequence)
    elif kind == "append":
        c["new"] = _log(rng, 40, 100000)
        c["batch"] = max(1, min(32, _log(rng, 1, 32), 400000 // c["new"]))
        c["context"] = rng.choice([0, _log(rng, 100, 16000)])
        if c["batch"] > 2 and rng.random() < 0.5:
            c["new_min"] = max(1, c["new"] // 6)
    else:
        c["new"] = _log(rng, 24, 6000)
        c["context"] = rng.choice([0, _log(rng, 100, 30000)])
        cost = c["new"] * (c["context"] + c["new"] + 4000) * hkv * group
        c["batch"] = max(1, min(4, _log(rng, 1, 4), (8192 * 12288 * 32) // (2 * cost)))
        while c["batch"] * c["new"] * (c["context"] + c["new"] + 4000) * hkv * group > 8192 * 12288 * 32 // 2:
            c["new"] = c["new"] * 2 // 3
    return _case(**c)


def _room(case):
    """Passes that a slot takes before it is rewound: a prompt fills it, a turn or a chunk leaves space for more."""
    if case["kind"] == "decode":
        return DECODE_ROOM
    return 1 if case["context"] == 0 else 8


def _workload(case, seed):
    return synth.Workload("case", int(seed), batch=case["batch"], n_q_heads=case["hq"], n_kv_heads=case["hkv"],
                          head_dim=case["d"], block_size=case["block"], top_k=case["top_k"], context=max(case["context"], 1),
                          context_min=case["context_min"], kv_dtype=case["dtype"], n_needles=case["needles"],
                          n_outlier_channels=case["outliers"], drift_step=case["drift"],
                          n_steps=_room(case) * case["new"])


def _chunk(case, w, seed):
    """K and V of `new` tokens per sequence, and the queries of all their positions."""
    g = torch.Generator(device=DEV).manual_seed((int(seed) * 7919 + 5) & 0x7FFFFFFF)
    shape = (w.batch, w.n_kv_heads, case["new"], w.head_dim)
    k = torch.randn(shape, generator=g, device=DEV)
    v = torch.randn(shape, generator=g, device=DEV)
    if w.n_outlier_channels:
        ch = torch.as_tensor(synth.outlier_channels(w), device=DEV)
        for h in range(w.n_kv_heads):
            k[:, h, :, ch[h]] *= w.outlier_scale
    q = None
    if case["kind"] == "prefill":
        q0 = synth.query_directions(w).to(DEV).repeat_interleave(w.group, dim=1)[:, None]
        q = torch.randn(w.batch, case["new"], w.n_q_heads, w.head_dim, generator=g, device=DEV)
        q = ((q0 + 0.5 * q) / math.sqrt(1.25)).to(w.torch_dtype)
    return k.to(w.torch_dtype), v.to(w.torch_dtype), q


def prepare(case, seed):
    w = _workload(case, seed)
    flags = binding.SPLA_STATS_BF16 if case["stats16"] else 0
    cache = binding.SplaCache(runner.config_for(w, flags=flags, window=(case["window"], case["stride"]) if case["window"] else None), DEV)
    cache.bufs.k_cache.zero_()
    cache.bufs.v_cache.zero_()
    s = dict(case=case, cache=cache, gamma=synth.gamma(w).to(DEV), room=_room(case), left=_room(case), step=0)
    if case["context"]:
        K, V, lens = runner.generate_prefill(w, DEV)
        cache.append_tokens(K, V, lens if case["context_min"] else None)
        del K, V
    s["bound"] = int(cache.bufs.seq_lens.max().item())
    s["lens"], s["state"] = cache.bufs.seq_lens.clone(), cache.bufs.rla_state.clone()
    cache.set_length_bound(s["bound"])
    dev = dict(device=DEV)
    if case["kind"] == "decode":
        s["q"] = [synth.step_queries(w, i, DEV) for i in range(4)]
        s["kv"] = [synth.step_kv(w, i, DEV) for i in range(4)]
        s["out"] = torch.empty(w.batch, w.n_q_heads, w.head_dim, dtype=torch.float32, **dev)
        s["sel"] = cache.new_sel_buffer()
    else:
        s["k"], s["v"], s["q"] = _chunk(case, w, seed)
        s["n_new"] = None
        if case["new_min"]:
            g = torch.Generator().manual_seed(int(seed) & 0x7FFFFFFF)
            s["n_new"] = torch.randint(case["new_min"], case["new"] + 1, (w.batch,), generator=g, dtype=torch.int32).to(DEV)
        if case["kind"] == "prefill":
            s["out"] = torch.empty(w.batch, case["new"], w.n_q_heads, w.head_dim, dtype=torch.float32, **dev)
            s["sel"] = torch.empty(w.batch, case["new"], w.n_kv_heads, w.top_k, dtype=torch.int32, **dev)
    return s


def run(s):
    c, b = s["cache"], s["cache"].bufs
    if s["left"] == 0:                                    # the slot is full: back to the context it began with
        b.seq_lens.copy_(s["lens"])
        b.rla_state.copy_(s["state"])
        c.set_length_bound(s["bound"])
        s["left"] = s["room"]
    s["left"] -= 1
    kind = s["case"]["kind"]
    after = [b.seq_lens, b.rla_state, b.stats, b.tok_lse]
    if kind == "decode":
        i = s["step"] = (s["step"] + 1) % 4
        k, v = s["kv"][i]
        c.append_decode(k, v, s["q"][i], s["gamma"], out=s["out"], sel_idx=s["sel"])
        return [s["out"], s["sel"]] + after
    if kind == "append":
        c.append_tokens(s["k"], s["v"], s["n_new"])
        return after + [b.k_cache, b.v_cache]
    c.prefill(s["k"], s["v"], s["q"], s["gamma"], out=s["out"], sel_idx=s["sel"])
    return [s["out"], s["sel"]] + after + [b.k_cache, b.v_cache]


def work(case):
    """What one pass cannot do without, at the mean length and the context that a slot begins with."""
    e = 2 if case["dtype"] == "bf16" else 4
    d, B, G = case["d"], case["block"], case["hq"] // case["hkv"]
    U = case["batch"] * case["hkv"]
    L0 = (case["context"] + case["context_min"]) / 2 if case["context_min"] else case["context"]
    n = (case["new"] + case["new_min"]) / 2 if case["new_min"] else case["new"]
    windows = (B - case["window"]) // case["stride"] + 1 if case["window"] else 1
    rec = windows * 2 * d * (2 if case["stats16"] else 4)
    state = d * d * 4
    # the tokens go in: read and written once, a log-sum-exp each, the records of the blocks they touch, the state in and out
    touched = math.ceil(n / B)
    bytes_ = U * (4 * n * d * e + 4 * n + touched * rec + 2 * state)
    flops = U * (2 * n * d * d + 6 * n * d)
    if case["kind"] == "append":
        return {"bytes": bytes_, "flops": flops}
    row_io = case["batch"] * n * case["hq"] * d * (e + 4)          # queries in, outputs out
    if case["kind"] == "decode":
        nblk = math.ceil((L0 + 1) / B)
        picked = min(case["top_k"], nblk)
        bytes_ += row_io + U * (nblk * rec + picked * B * (2 * d * e + 4))
        flops += U * G * (4 * d * windows * nblk + 8 * d * picked * B + 2 * d * d)
        return {"bytes": bytes_, "flops": flops}
    # prefill: position t sees (L0 + t) / B blocks; what lies before the chunk is read once (no more of K and V than is picked)
    tot = pick = 0.0
    for i in range(64):
        nblk = math.ceil((L0 + (i + 0.5) / 64 * n) / B)
        tot += nblk * n / 64
        pick += min(case["top_k"], nblk) * n / 64
    old = math.ceil(L0 / B)
    bytes_ += row_io + U * (old * rec + min(old, pick) * B * (2 * d * e + 4))
    flops += U * G * (4 * d * tot + 8 * d * pick * B + 2 * n * d * d)
    return {"bytes": bytes_, "flops": flops}


def tolerance(case):
    """Measured against the library's general kernels (`SPLA_GENERAL_KERNELS`: fp32 sums in another order), a chunk
    against the same tokens decoded one at a time; about four times what was seen.

    Appends: K/V bit for bit, the state 5.7e-6 (largest 1e-4); summaries in 16 bits may round the other way.  fp32
    attention: 6e-8.  bf16 attention: 4e-4 to 7e-4 (largest 6e-3), from the probabilities' 8 bits.  No selection
    differed; log masses that are 1e-5 off change 1 in 3000 of them, where the k-th and the next score tie, and with
    it that position's output, by a good part of its size.
    """
    if case["kind"] == "append":
        return {"rel": 3e-4, "max": 1e-2} if case["stats16"] else {"rel": 3e-5, "max": 6e-4}
    ties = {"max": 0.5, "differ": 5e-4 if case["kind"] == "prefill" else 5e-3}
    return dict(ties, rel=1e-5 if case["dtype"] == "f32" else 3e-3)
