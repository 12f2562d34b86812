"""Measured cases of the decode step: the calls that a program using this package
makes, over the sizes it makes them with.

Every case is a dict of plain values whose ``kind`` names the entry points:

* ``step``  the first decode step of a batch of prompts: gate states and row mask
  reset, then ``rgd_decode_step`` (attention, then the sample head with the gate).
* ``loop``  a whole gated generation captured as one CUDA graph
  (``device.DeviceLoop``), replayed.
* ``attn``  ``rgd_prefix_decode_attn`` alone, as a model calls it per layer.
* ``head``  ``rgd_sample_head`` alone (logits-only callers).
* ``soft``  one probe step of ``rgd_soft_gate``.
* ``gate``  ``rgd_residual_precheck`` and ``rgd_probe_gate`` for probe tokens that
  were decoded elsewhere.

Inputs are drawn on the GPU from the seed: N(0, 1) queries and bf16 KV in 16-token
pages scattered over the pool, Zipf(1.1)-ranked log-probabilities plus N(0, 1) noise
as logits, random refusal sequences -- the package's synthetic workloads.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2607_20791_gb300 import binding, device, workloads

PAGE = 16
DEV = "cuda"


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------
def _attn_fields(groups, rows, q_heads, kv_heads, dim, prompt_lo, prompt_hi, suffix):
    """prompt lengths run from prompt_lo to prompt_hi (log-uniform), suffixes from 0 to `suffix`."""
    return {"groups": groups, "rows": rows, "q_heads": q_heads, "kv_heads": kv_heads, "dim": dim,
            "prompt_lo": prompt_lo, "prompt_hi": prompt_hi, "suffix": suffix}


def _head_fields(vocab, dtype, sampling):
    return {"vocab": vocab, "dtype": dtype, "sampling": sampling}


def listed():
    return [
        # one short prompt, small heads and vocabulary: a unit-test-sized model or a
        # draft model; launches and latency are all there is
        {"name": "step_tiny", "kind": "step", "masked": 0.0, "seqs": 8,
         **_attn_fields(1, 3, 4, 1, 64, 128, 128, 16), **_head_fields(4096, "f32", "usual")},
        # the ordinary serving step: 16 prompts of 512-2048 tokens, 1 probe and 4 samples each
        {"name": "step_8b", "kind": "step", "masked": 0.0, "seqs": 64,
         **_attn_fields(16, 5, 32, 8, 128, 512, 2048, 256), **_head_fields(128256, "f32", "usual")},
        # high-batch serving: 256 prompts, 1 probe and 1 sample each, 30 % of the samples masked
        {"name": "step_high_batch", "kind": "step", "masked": 0.3, "seqs": 64,
         **_attn_fields(256, 2, 32, 8, 128, 128, 8192, 256), **_head_fields(152064, "bf16", "wide")},
        # the gated generation of a batch from the prompt end: 128 steps in one graph
        {"name": "loop_8b", "kind": "loop", "steps": 128, "seqs": 64,
         **_attn_fields(16, 5, 32, 8, 128, 512, 2048, 0), **_head_fields(128256, "f32", "usual")},
        # a single request's attention: little KV for the whole chip
        {"name": "attn_single", "kind": "attn", "masked": 0.0, **_attn_fields(1, 5, 32, 8, 128, 3000, 3000, 200)},
        # more samples per prompt (36 queries per kv head), ragged lengths
        {"name": "attn_samples", "kind": "attn", "masked": 0.1, **_attn_fields(12, 9, 32, 8, 128, 500, 6000, 500)},
        # long prompts: 4 x 32768 tokens, 72 queries per kv head
        {"name": "attn_long", "kind": "attn", "masked": 0.0, **_attn_fields(4, 9, 64, 8, 128, 32768, 32768, 1024)},
        # a handful of rows over an odd vocabulary (rows off 16-byte boundaries), kept mask wanted
        {"name": "head_odd", "kind": "head", "rows": 8, "mask": True, **_head_fields(32001, "f32", "usual")},
        # a serving batch of bf16 logits
        {"name": "head_bf16", "kind": "head", "rows": 256, "mask": False, **_head_fields(128256, "bf16", "sweep")},
        # the largest head: 1 GB of fp32 logits
        {"name": "head_large", "kind": "head", "rows": 1024, "mask": False, **_head_fields(262144, "f32", "sweep")},
        # the soft gate's probe step on the probe rows of a 16 x 5 step
        {"name": "soft_gate", "kind": "soft", "groups": 16, "rows": 5, "seqs": 64, "top_k": 40,
         **_head_fields(128256, "f32", "usual")},
        # prechecks and 32-token probes of 1024 prompts against 1000 refusal sequences
        {"name": "gate", "kind": "gate", "groups": 1024, "rows": 2, "seqs": 1000, "tokens": 32, "d": 4096,
         "vocab": 128256, "dtype": "bf16"},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


HEADS = ((4, 1, 64), (8, 2, 64), (32, 8, 64), (16, 16, 128), (28, 4, 128), (32, 8, 128), (64, 8, 128))


def _draw_attn(rng, token_bytes_cap):
    hq, hkv, dim = rng.choice(HEADS)
    rows = rng.randint(1, min(16, 128 // (hq // hkv)))
    groups = _log(rng, 1, 256)
    cap = max(32, token_bytes_cap // (groups * hkv * dim * 4))  # tokens per group
    hi = min(32768, cap, _log(rng, 16, 32768))
    lo = rng.randint(1, hi)
    return _attn_fields(groups, rows, hq, hkv, dim, lo, hi, rng.randint(0, min(1024, max(1, cap // rows))))


def _draw_head(rng, rows, cap_bytes):
    dtype = rng.choice(("f32", "bf16"))
    hi = min(262144, max(1000, cap_bytes // (rows * (4 if dtype == "f32" else 2))))
    vocab = _log(rng, 1000, hi)
    if rng.random() < 0.5:
        vocab = (vocab + 7) // 8 * 8
    return _head_fields(vocab, dtype, "sweep" if rows >= 200 and rng.random() < 0.5 else "usual")


def draw(rng):
    kind = rng.choice(("step", "step", "attn", "attn", "head", "head", "loop", "soft", "gate"))
    if kind in ("step", "attn"):
        c = {"kind": kind, "masked": rng.choice((0.0, 0.0, 0.1, 0.3)), **_draw_attn(rng, 600 << 20)}
        if kind == "step":
            c.update(seqs=_log(rng, 1, 1000), **_draw_head(rng, c["groups"] * c["rows"], 300 << 20))
        return c
    if kind == "head":
        rows = _log(rng, 1, 1024)
        c = {"kind": kind, "rows": rows, **_draw_head(rng, rows, 1 << 30)}
        return {**c, "mask": c["vocab"] * rows < 1 << 24 and rng.random() < 0.3}
    if kind == "loop":
        c = {"kind": kind, "steps": rng.randint(2, 48), "seqs": _log(rng, 1, 200), **_draw_attn(rng, 64 << 20)}
        c.update(groups=min(c["groups"], 24), rows=max(2, min(c["rows"], 5)), suffix=0)
        return {**c, **_head_fields(_log(rng, 4000, 128256), "f32", "usual")}
    if kind == "soft":
        groups, rows = _log(rng, 1, 64), rng.randint(1, 6)
        return {"kind": kind, "groups": groups, "rows": rows, "seqs": _log(rng, 1, 600), "top_k": rng.randint(1, 100),
                **_head_fields(_log(rng, 4000, 262144), rng.choice(("f32", "bf16")), "usual")}
    return {"kind": "gate", "groups": _log(rng, 1, 4096), "rows": rng.randint(1, 6), "seqs": _log(rng, 1, 2000),
            "tokens": _log(rng, 1, 64), "d": _log(rng, 64, 8192), "vocab": _log(rng, 4000, 262144),
            "dtype": rng.choice(("f32", "bf16"))}


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _gen(seed, salt):
    g = torch.Generator(device=DEV)
    g.manual_seed((int(seed) * 1000003 + salt) & 0x7FFFFFFFFFFFFFFF)
    return g


def _np_rng(seed, salt):
    return np.random.default_rng([int(seed) & 0x7FFFFFFF, salt])


def _lengths(c, seed):
    rng = _np_rng(seed, 1)
    G, R = c["groups"], c["groups"] * c["rows"]
    plen = np.round(np.exp(rng.uniform(math.log(c["prompt_lo"]), math.log(c["prompt_hi"]), G))).astype(np.int32)
    slen = rng.integers(0, c["suffix"] + 1, R).astype(np.int32)
    active = np.ones(R, np.uint8)
    if c.get("masked") and c["rows"] > 1:
        off = rng.permutation(G)[: int(round(c["masked"] * G))]
        for g in off:  # a group gated off after its probe: only the probe row goes on
            active[g * c["rows"] + 1:(g + 1) * c["rows"]] = 0
    return plen, slen, active


def _tables(c, seed, room=0):
    plen, slen, active = _lengths(c, seed)
    pp, sp = (plen + PAGE - 1) // PAGE, (slen + room + PAGE - 1) // PAGE
    num_pages = int(pp.sum() + sp.sum()) + 3
    perm = _np_rng(seed, 2).permutation(num_pages).astype(np.int32)
    pbt = np.full((c["groups"], max(1, int(pp.max()))), -1, np.int32)
    sbt = np.full((len(slen), max(1, int(sp.max()))), -1, np.int32)
    at = 0
    for table, counts in ((pbt, pp), (sbt, sp)):
        for i, n in enumerate(counts):
            table[i, :n] = perm[at:at + n]
            at += n
    return plen, slen, active, pbt, sbt, num_pages


def _kv(c, seed, num_pages):
    shape = (num_pages, c["kv_heads"], PAGE, c["dim"])
    return tuple(torch.randn(shape, generator=_gen(seed, 10 + i), device=DEV, dtype=torch.bfloat16) for i in range(2))


def _attn_case(c, seed, room=0):
    """The package's attention inputs (host arrays) and the KV pools (on the GPU)."""
    plen, slen, active, pbt, sbt, num_pages = _tables(c, seed, room)
    R = c["groups"] * c["rows"]
    q = torch.randn((R, c["q_heads"], c["dim"]), generator=_gen(seed, 12), device=DEV, dtype=torch.bfloat16)
    case = workloads.AttnCase(
        name="case", num_groups=c["groups"], rows_per_group=c["rows"], num_q_heads=c["q_heads"],
        num_kv_heads=c["kv_heads"], head_dim=c["dim"], q=q.view(torch.int16).cpu().numpy().view(np.uint16),
        k_pages=None, v_pages=None, num_pages=num_pages, prompt_block_table=pbt, prompt_len=plen,
        suffix_block_table=sbt, suffix_len=slen, row_active=active, softmax_scale=1.0 / math.sqrt(c["dim"]))
    return case, _kv(c, seed, num_pages)


def _logits(rows, vocab, dtype, seed):
    base = -1.1 * torch.log(torch.arange(1, vocab + 1, dtype=torch.float64))
    base = (base - torch.logsumexp(base, 0)).float().to(DEV)
    gen = _gen(seed, 20)
    out = torch.empty((rows, vocab), dtype=torch.float32 if dtype == "f32" else torch.bfloat16, device=DEV)
    for r in range(rows):
        perm = torch.randperm(vocab, generator=gen, device=DEV)
        out[r] = base[perm] + torch.randn(vocab, generator=gen, device=DEV)
    return out


def _sampling(rows, rpg, sampling, seed):
    """Temperatures, min-p and seeds per row; rpg > 0: every group's first row is a greedy probe."""
    rng = _np_rng(seed, 3)
    i = np.arange(rows)
    if sampling == "sweep":
        t, p = np.array([0.0, 1.0, 2.0, 5.0, 10.0])[i % 5], np.array([0.0, 0.05, 0.1, 0.3])[(i // 5) % 4]
    elif sampling == "wide":
        t, p = rng.uniform(0.7, 5.0, rows), rng.uniform(0.0, 0.2, rows)
    else:
        t, p = np.array([1.0, 1.5, 2.0, 3.0])[i % 4], np.array([0.05, 0.1])[i % 2]
    probe = (i % rpg == 0) if rpg else np.zeros(rows, bool)
    t = np.where(probe, 0.0, t)
    seeds = rng.integers(0, np.iinfo(np.uint64).max, size=rows, dtype=np.uint64)
    return probe.astype(np.uint8), t.astype(np.float32), p.astype(np.float32), seeds


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to(DEV)


class State:
    pass


def _head_state(s, c, rows, rpg, seed, mask=False):
    probe, t, p, seeds = _sampling(rows, rpg, c["sampling"], seed)
    s.logits = _logits(rows, c["vocab"], c["dtype"], seed)
    s.probe, s.temp, s.minp, s.seeds = _dev(probe), _dev(t), _dev(p), _dev(seeds.view(np.int64))
    s.token = torch.zeros(rows, dtype=torch.int32, device=DEV)
    s.kept = torch.zeros(rows, dtype=torch.int32, device=DEV)
    s.mask = torch.zeros((rows, c["vocab"]), dtype=torch.uint8, device=DEV) if mask else None


def _gate_state(s, c, seed, seqs, rows):
    s.trie = binding.Trie(seqs, 2)
    s.state = binding.new_gate_state(c["groups"])
    s.groups, s.rows = c["groups"], rows


def prepare(c, seed):
    s = State()
    s.kind = kind = c["kind"]
    s.status = torch.zeros(1, dtype=torch.int32, device=DEV)
    if kind in ("step", "attn"):
        case, kv = _attn_case(c, seed)
        s.att = device.attn_to_device(case, kv=kv)
        s.att.lse.zero_()
    if kind == "step":
        R = c["groups"] * c["rows"]
        _head_state(s, c, R, c["rows"], seed)
        seqs = workloads.make_refusal_set(c["seqs"], 2, 8, c["vocab"], seed & 0x7FFFFFFF)
        _gate_state(s, c, seed, seqs, c["rows"])
        s.active0 = s.att.row_active.clone()  # the rows that decode at this step
        s.active = s.att.row_active
    elif kind == "loop":
        s.loop = _loop(c, seed)
    elif kind == "head":
        _head_state(s, c, c["rows"], 0, seed, c["mask"])
        s.step = seed & 0xFFFF
    elif kind == "soft":
        s.c = c
        s.seqs, s.eos, s.rho = _soft_setting(c, seed)
        R = c["groups"] * c["rows"]
        s.logits = _logits(R, c["vocab"], c["dtype"], seed)
        _plant(s.logits, c, s.seqs, seed)
        _gate_state(s, c, seed, s.seqs, c["rows"])
        s.active = torch.ones(R, dtype=torch.uint8, device=DEV)
        s.token = torch.zeros(c["groups"], dtype=torch.int32, device=DEV)
        s.mass = torch.zeros(c["groups"], dtype=torch.float32, device=DEV)
    elif kind == "gate":
        s.c = c
        h, w, s.bias, s.theta = _precheck_inputs(c, seed)
        s.h, s.w = h, w
        seqs = workloads.make_refusal_set(c["seqs"], 2, 12, c["vocab"], seed & 0x7FFFFFFF)
        s.tokens = _dev(workloads.make_probe_streams(seqs, c["groups"], c["tokens"], c["vocab"], seed & 0x7FFFFFFF))
        _gate_state(s, c, seed, seqs, c["rows"])
        s.active = torch.ones(c["groups"] * c["rows"], dtype=torch.uint8, device=DEV)
        s.prob = torch.zeros(c["groups"], dtype=torch.float32, device=DEV)
    return s


def _loop_inputs(c, seed):
    """Refusal sequences, stop token and planted probe streams of a generation."""
    vocab, s31 = c["vocab"], seed & 0x7FFFFFFF
    eos = vocab - 1
    seqs = workloads.make_refusal_set(c["seqs"], 2, 8, vocab, s31, avoid=[eos])
    return seqs, eos, workloads.loop_probe_streams(seqs, c["groups"], c["steps"], vocab, s31, eos)


def _loop(c, seed):
    case, kv = _attn_case(c, seed, room=c["steps"])
    R = c["groups"] * c["rows"]
    probe, t, p, seeds = _sampling(R, c["rows"], c["sampling"], seed)
    head = workloads.HeadCase(name="loop", logits=_logits(R, c["vocab"], c["dtype"], seed).cpu().numpy(), dtype="f32",
                              is_probe=probe, temperature=t, min_p=p, seed=seeds, step=0,
                              row_active=np.ones(R, np.uint8))
    seqs, eos, streams = _loop_inputs(c, seed)
    lc = workloads.LoopCase(name="loop", attn=case, head=head, refusal_seqs=seqs, probe_streams=streams, eos=eos,
                            max_len=c["steps"], gate_cap=3, n_steps=c["steps"])
    loop = device.DeviceLoop(lc, torch.cuda.Stream(), keep_history=False, kv=kv)
    torch.cuda.synchronize()  # (the loop's buffers, before its own stream uses them)
    loop.capture()
    return loop


def _soft_setting(c, seed):
    vocab = c["vocab"]
    eos = vocab - 1
    return workloads.make_refusal_set(c["seqs"], 2, 8, vocab, seed & 0x7FFFFFFF, avoid=[eos]), eos, 0.05


def _plant(logits, c, seqs, seed):
    """In two groups of three, first tokens of some refusal sequences lie a little below the row's maximum."""
    rng = _np_rng(seed, 5)
    for g in range(c["groups"]):
        if g % 3 == 0:
            continue
        row = logits[g * c["rows"]]
        top = float(row.max())
        for _ in range(3):
            row[int(seqs[int(rng.integers(len(seqs)))][0])] = top - float(rng.uniform(0.2, 3.0))


def _precheck_inputs(c, seed):
    h = torch.randn((c["groups"], c["d"]), generator=_gen(seed, 30), device=DEV)
    h = h if c["dtype"] == "f32" else h.to(torch.bfloat16)
    w = torch.randn(c["d"], generator=_gen(seed, 31), device=DEV) * (8.0 / math.sqrt(c["d"]))
    return h, w, -2.0, 1e-5


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
MAX_LEN, EOS = 128, -1


def run(s):
    if s.kind == "attn":
        s.att.run()
        return {"out": s.att.out, "lse": s.att.lse, "status": s.att.dev_status}
    if s.kind == "step":
        a = s.att
        binding.rgd_gate_state_init(s.state, s.groups)
        s.active.copy_(s.active0)
        binding.rgd_decode_step(a.shape, a.q, a.k_pages, a.v_pages, a.prompt_block_table, a.prompt_len,
                                a.suffix_block_table, a.suffix_len, a.softmax_scale, a.out, a.lse, a.workspace,
                                s.logits, s.probe, s.temp, s.minp, s.seeds, 0, s.active, s.token, s.kept, s.trie,
                                EOS, MAX_LEN, s.state, s.status)
        return {"out": a.out, "lse": a.lse, "token": s.token, "kept": s.kept, "state": s.state, "active": s.active,
                "status": s.status}
    if s.kind == "loop":
        s.loop.graph.replay()
        return {"out": s.loop.att.out, "token": s.loop.tok, "state": s.loop.state, "active": s.loop.row_active,
                "suffix": s.loop.suffix_len, "status": s.loop.status}
    if s.kind == "head":
        binding.rgd_sample_head(s.logits, s.probe, s.temp, s.minp, s.seeds, s.step, None, s.token, s.kept, s.mask,
                                s.status)
        return {"token": s.token, "kept": s.kept, "mask": s.mask, "status": s.status}
    if s.kind == "soft":
        c = s.c
        binding.rgd_gate_state_init(s.state, s.groups)
        s.active.fill_(1)
        binding.rgd_soft_gate(s.trie, s.groups, s.rows, s.logits, s.rows * c["vocab"], c["top_k"], s.rho, 3, s.eos,
                              MAX_LEN, s.state, s.token, s.active, s.mass, s.status)
        return {"token": s.token, "mass": s.mass, "state": s.state, "active": s.active, "status": s.status}
    c = s.c
    binding.rgd_gate_state_init(s.state, s.groups)
    s.active.fill_(1)
    binding.rgd_residual_precheck(s.h, s.w, s.bias, s.theta, s.rows, s.state, s.active, s.prob, s.status)
    binding.rgd_probe_gate(s.trie, s.groups, s.rows, s.tokens, c["tokens"], c["tokens"], EOS, MAX_LEN, s.state,
                           s.active, s.status)
    return {"prob": s.prob, "state": s.state, "active": s.active, "status": s.status}


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def _attn_work(c, steps=0):
    """Expected bytes and operations of one attention call (`steps`: the mean over a loop's growing suffixes)."""
    G, rpg, hq, hkv, D = c["groups"], c["rows"], c["q_heads"], c["kv_heads"], c["dim"]
    lo, hi = c["prompt_lo"], c["prompt_hi"]
    prompt = lo if lo == hi else (hi - lo) / math.log(hi / lo)
    suffix = steps / 2 if steps else c["suffix"] / 2
    rows = G * (rpg - (rpg - 1) * c.get("masked", 0.0))
    tokens = G * prompt + rows * suffix
    byt = tokens * hkv * D * 4 + rows * hq * D * 4 + rows * hq * 4
    return byt, 4.0 * rows * hq * D * (prompt + suffix)


def work(c):
    kind = c["kind"]
    es = 4 if c.get("dtype") == "f32" else 2
    if kind == "attn":
        b, f = _attn_work(c)
    elif kind == "step":
        b, f = _attn_work(c)
        rows = c["groups"] * (c["rows"] - (c["rows"] - 1) * c["masked"])
        b, f = b + rows * (c["vocab"] * es + 8), f + rows * c["vocab"] * 2.0
    elif kind == "loop":
        # about half the rows of a group stay active once its gate has decided
        b, f = _attn_work(c, c["steps"])
        rows = 0.5 * c["groups"] * c["rows"]
        b, f = c["steps"] * (b + rows * c["vocab"] * es), c["steps"] * (f / 2 + rows * c["vocab"] * 2.0)
    elif kind == "head":
        b = c["rows"] * (c["vocab"] * (es + (1 if c["mask"] else 0)) + 8)
        f = c["rows"] * c["vocab"] * 2.0
    elif kind == "soft":
        b, f = c["groups"] * (c["vocab"] * es + 48), c["groups"] * c["vocab"] * 2.0
    else:
        b = c["groups"] * (c["d"] * es + c["tokens"] * 4 + 44 + 2 * c["rows"]) + c["d"] * 4
        f = c["groups"] * c["d"] * 2.0
    return {"bytes": float(b), "flops": float(f)}


def tolerance(c):
    """Attention: bf16 outputs (one rounding is 2^-9 of the value; an output is a few units of 1e-3 from
    the 64-bit result), 32-bit log-sum-exps.  Tokens: draws within the 32-bit sums' rounding of a step of
    the distribution function may fall to either side.  The gates' masses and probabilities are 32-bit sums,
    1e-7 from the 64-bit ones."""
    if c["kind"] in ("attn", "step", "loop"):
        return {"rel": 7e-3, "max": 3e-2, "differ": 0.01}
    if c["kind"] == "head":
        return {"rel": 0.0, "differ": 0.01}
    return {"rel": 2e-6, "max": 2e-5, "differ": 0.01}


# ---------------------------------------------------------------------------
# the same in 64 bits
# ---------------------------------------------------------------------------
def _exact_attn(c, seed, active, slen, room=0):
    plen, _, _, pbt, sbt, num_pages = _tables(c, seed, room)
    k, v = _kv(c, seed, num_pages)
    G, rpg, hq, hkv, D = c["groups"], c["rows"], c["q_heads"], c["kv_heads"], c["dim"]
    gq = hq // hkv
    q = torch.randn((G * rpg, hq, D), generator=_gen(seed, 12), device=DEV, dtype=torch.bfloat16).double()
    out = torch.zeros((G * rpg, hq, D), dtype=torch.float64, device=DEV)
    lse = torch.zeros((G * rpg, hq), dtype=torch.float64, device=DEV)

    def tokens(pool, table, n):  # [hkv, n, D]
        pages = torch.from_numpy(table[: (n + PAGE - 1) // PAGE].astype(np.int64)).to(DEV)
        return pool[pages].permute(1, 0, 2, 3).reshape(hkv, -1, D)[:, :n].double()

    scale = 1.0 / math.sqrt(D)
    for g in range(G):
        kp, vp = tokens(k, pbt[g], int(plen[g])), tokens(v, pbt[g], int(plen[g]))
        for r in range(g * rpg, (g + 1) * rpg):
            if not active[r]:
                continue
            kk, vv = kp, vp
            qr = q[r].reshape(hkv, gq, D)
            sp = qr @ kk.transpose(1, 2) * scale
            ks, vs = tokens(k, sbt[r], int(slen[r])), tokens(v, sbt[r], int(slen[r]))
            ss = qr @ ks.transpose(1, 2) * scale
            both = torch.cat([sp, ss], 2)
            l = torch.logsumexp(both, 2, keepdim=True)
            w = torch.exp(both - l)
            n = sp.shape[2]
            out[r] = (w[:, :, :n] @ vv + w[:, :, n:] @ vs).reshape(hq, D)
            lse[r] = l.reshape(hq)
    return out, lse


def _loop_last_active(c, seed):
    """The last step at which each row decodes: its group's probe matched by a plain scan of the sequences."""
    seqs, eos, streams = _loop_inputs(c, seed)
    n, rpg = c["steps"], c["rows"]
    last = np.full(c["groups"] * rpg, n - 1, np.int32)
    for g in range(c["groups"]):
        q, confirmed, done, refused = [], False, n - 1, None
        for t in range(n):
            y = int(streams[g, t])
            if y == eos:
                done, refused = t, (t if refused is None else refused)
                break
            q.append(y)
            if not confirmed:
                if any(len(s) >= 2 and list(s) == q[: len(s)] for s in seqs):
                    confirmed, refused = True, t
                elif not any(list(s[: len(q)]) == q for s in seqs):
                    done = t
                    break
            if len(q) >= n:
                done, refused = t, (t if refused is None else refused)
                break
        last[g * rpg] = done
        if refused is not None:
            last[g * rpg + 1:(g + 1) * rpg] = refused
    return last


def exact(c, seed):
    kind = c["kind"]
    if kind == "attn":
        _, slen, active = _lengths(c, seed)
        out, lse = _exact_attn(c, seed, active, slen)
        return {"out": out, "lse": lse, "status": None}
    if kind == "step":
        _, slen, active = _lengths(c, seed)
        out, lse = _exact_attn(c, seed, active, slen)
        return {"out": out, "lse": lse, "token": None, "kept": None, "state": None, "active": None, "status": None}
    if kind == "loop":
        # a row's last output: its prompt and the tokens appended before its last active step
        last = _loop_last_active(c, seed)
        out, _ = _exact_attn(c, seed, np.ones(len(last), np.uint8), last, room=c["steps"])
        return {"out": out, "token": None, "state": None, "active": None, "suffix": None, "status": None}
    if kind == "soft":
        seqs, eos, _ = _soft_setting(c, seed)
        logits = _logits(c["groups"] * c["rows"], c["vocab"], c["dtype"], seed)
        _plant(logits, c, seqs, seed)
        mass = torch.full((c["groups"],), -1.0, dtype=torch.float64)
        first = sorted({int(s[0]) for s in seqs} | {eos})
        for g in range(c["groups"]):
            row = logits[g * c["rows"]].double().cpu().numpy()
            order = np.lexsort((np.arange(len(row)), -row))  # larger first, then the lower index
            if int(order[0]) in first:
                continue
            prob = np.exp(row - row.max())
            top = set(order[: c["top_k"]].tolist())
            mass[g] = float(sum(prob[a] for a in first if a in top) / prob.sum())
        return {"token": None, "mass": mass.to(DEV), "state": None, "active": None, "status": None}
    if kind == "gate":
        h, w, bias, _ = _precheck_inputs(c, seed)
        return {"prob": torch.sigmoid(h.double() @ w.double() + bias), "state": None, "active": None, "status": None}
    return None  # the head gives whole numbers only
