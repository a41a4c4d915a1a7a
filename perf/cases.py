"""The calls whose time matters to a user of libism, with their inputs.

Four kinds of call, each through the package's public entry points:

  train    one attention layer of a training step: forward and backward over
           packed dialogues (``ism.fwd`` / ``ism.bwd`` or the rotary pair),
           returning O, LSE and the gradients
  forward  the one-pass forward on e4m3 inputs (``ism.fwd_e4m3``): scoring or
           prefilling whole dialogues
  append   a new turn of a dialogue against its KV cache
           (``ism.prefill_append*``): time to first token
  decode   a short answer generated token by token against the KV cache
           (``ism.AppendStep`` or ``ism.prefill_append*``): time per token

Dialogue structures (turns, query and answer lengths) and cache lengths come
from the case alone; the values come from the seed.
"""
import math

import numpy as np
import torch

from paper_2408_00539_gb300 import ism
from paper_2408_00539_gb300 import workloads as wl

DEVICE = "cuda"
PAGE = 256  # rows of a cache page

#: A case is one of these with some fields replaced.
#:   seqs, tokens   packed dialogues and their tokens together; "even" lengths or "random" cut points
#:   turns          most turns of a dialogue (at least 2)
#:   plan           "none": every call builds its metadata; "step": a plan built in each pass, as a training
#:                  step of one layer does; "kept": a plan built beforehand, as the later layers of a step see it
#:   batch, cache   sequences of an append or a decode, and the longest one's cached tokens
#:   ragged         the sequences' cached lengths are spread over [cache / 16, cache]
#:   new            tokens appended in one call (append), or generated one by one (decode)
#:   layout         structure seed
_BASE = dict(kind="train", dtype="bf16", head_dim=128, hq=32, hkv=8, rope=False, layout=1,
             seqs=1, tokens=0, even=True, turns=16, plan="none", min_workspace=False,
             batch=0, cache=0, ragged=False, paged=False, new=0, query=True)


def _case(name=None, **fields):
    c = dict(_BASE, **fields)
    return dict(name=name, **c) if name else c


def listed():
    return [
        # The smallest training step: one 256-token dialogue, 2 heads of 64 in fp32 (the tiny configuration
        # of the tests): debugging a model, or a gradient check.
        _case("train_fp32_tiny", dtype="fp32", head_dim=64, hq=2, hkv=2, tokens=256, turns=3),
        # A small model's layer: 16 heads of 64, three dialogues of unequal, odd lengths.
        _case("train_d64_ragged", head_dim=64, hq=16, hkv=16, seqs=3, tokens=6001, even=False, layout=2),
        # The benchmark's step: two 8192-token dialogues, grouped-query heads, plan built once a step.
        _case("train_gqa_8k", seqs=2, tokens=16384, layout=3, plan="step"),
        # Multi-head attention (a KV head for each query head) at a medium length, calls without a plan.
        _case("train_mha_4k", hkv=32, seqs=4, tokens=16384, turns=8, layout=2),
        # Many short dialogues in one buffer, off every tile boundary, with rotary encoding: the middle layers
        # of a fine-tuning step.
        _case("train_short_rope", seqs=24, tokens=16001, even=False, turns=8, layout=4, rope=True, plan="kept"),
        # A long dialogue with the smallest backward workspace.
        _case("train_long_32k", tokens=32768, turns=100, layout=131, min_workspace=True),
        # Scoring whole dialogues in e4m3.
        _case("forward_e4m3_8k", kind="forward", dtype="e4m3", seqs=2, tokens=16384, layout=3),
        # One user's next short question late in a long session: the latency of a turn.
        _case("append_turn_40", kind="append", batch=1, cache=3000, new=40),
        # A batch of long contexts, each with a 512-token query.
        _case("append_16k_512", kind="append", batch=8, cache=16384, new=512),
        # One user's answer, token by token, with rotary encoding.
        _case("decode_single", kind="decode", batch=1, cache=3001, new=8, rope=True),
        # A serving batch of sessions of all lengths on a paged cache.
        _case("decode_paged_40", kind="decode", batch=40, cache=4000, new=8, ragged=True, paged=True),
        # A batch of long contexts on e4m3 caches.
        _case("decode_e4m3_16k", kind="decode", dtype="e4m3", batch=8, cache=16384, new=4),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["train", "train", "train", "forward", "append", "append", "decode", "decode"])
    layout = rng.randrange(1, 1 << 20)
    hq, hkv = rng.choice([(32, 8), (32, 8), (32, 32), (16, 4), (8, 2), (8, 8), (12, 4), (28, 4)])
    if kind == "train":
        dtype, d = rng.choice([("bf16", 128)] * 4 + [("bf16", 64), ("fp32", 64)])
        if dtype == "fp32":
            hq, hkv = rng.choice([(2, 2), (4, 2), (4, 4)])
        top = {("bf16", 128): 16384, ("bf16", 64): 8192, ("fp32", 64): 1024}[dtype, d]
        tokens = _log(rng, 64, top)
        return _case(dtype=dtype, head_dim=d, hq=hq, hkv=hkv, layout=layout, tokens=tokens,
                     seqs=min(_log(rng, 1, 32), max(1, tokens // 32)), even=False, turns=rng.choice([2, 4, 16]),
                     rope=rng.random() < 0.4, plan=rng.choice(["none", "step", "kept"]),
                     min_workspace=rng.random() < 0.25)
    if kind == "forward":
        tokens = _log(rng, 256, 16384)
        return _case(kind=kind, dtype="e4m3", hq=hq, hkv=hkv, layout=layout, tokens=tokens, even=False,
                     seqs=min(_log(rng, 1, 16), max(1, tokens // 64)), turns=rng.choice([2, 4, 16]))
    batch = _log(rng, 1, 40)
    cache = min(_log(rng, 100, 16384), 160000 // batch)
    dtype, rope, paged = rng.choice([("bf16", False, False), ("bf16", True, False), ("bf16", False, True),
                                     ("e4m3", False, False)])
    if kind == "append":
        return _case(kind=kind, dtype=dtype, hq=hq, hkv=hkv, layout=layout, batch=batch, cache=cache,
                     ragged=rng.random() < 0.5, rope=rope, paged=paged, new=min(_log(rng, 2, 1024), 8192 // batch),
                     query=rng.random() < 0.8)
    d = 64 if dtype == "bf16" and rng.random() < 0.15 else 128
    return _case(kind=kind, dtype=dtype, head_dim=d, hq=hq, hkv=hkv, layout=layout, batch=batch, cache=cache,
                 ragged=rng.random() < 0.5, rope=rope, paged=paged, new=rng.choice([4, 8]))


# ------------------------------------------------------------------ structure

def _segments(case):
    """The packed dialogues of a train or forward case (numpy)."""
    rng = np.random.Generator(np.random.PCG64(case["layout"]))
    n, total = case["seqs"], case["tokens"]
    if case["even"]:
        lens = [total // n + (i < total % n) for i in range(n)]
    else:  # cut points anywhere, at least 16 tokens each where that fits
        low = min(16, total // n)
        cuts = np.sort(rng.integers(0, total - n * low + 1, size=n - 1))
        lens = np.diff(np.concatenate([[0], cuts, [total - n * low]])) + low
    return wl.pack([wl.draw_dialogue(rng, int(x), 2, max(2, case["turns"])) for x in lens])


def _cache_lens(case):
    lens = np.full((case["batch"],), case["cache"], np.int32)
    if case["ragged"]:
        rng = np.random.Generator(np.random.PCG64(case["layout"]))
        lens = rng.integers(max(1, case["cache"] // 16), case["cache"] + 1, size=case["batch"]).astype(np.int32)
    return lens


def _ends(seg_end, seg_type):
    """The exclusive key bound of every row of one dialogue (numpy)."""
    out, start = [], 0
    for e, t in zip(seg_end, seg_type):
        e = int(e)
        out.append(np.full(e - start, e) if t == wl.QUERY else np.arange(start + 1, e + 1))
        start = e
    return np.concatenate(out).astype(np.int64)


def _visible(case):
    """Visible (row, key) pairs of one pass for one query head."""
    if case["kind"] in ("train", "forward"):
        s = _segments(case)
        return sum(int(_ends(se, st).sum()) for _, _, se, st in (s.seq(b) for b in range(s.num_seqs)))
    lens, n = _cache_lens(case).astype(np.int64), case["new"]
    own = n * n if case["kind"] == "append" and case["query"] else n * (n + 1) // 2
    return int(lens.sum()) * n + case["batch"] * own


# --------------------------------------------------------------------- inputs

def _bytes_of(dtype):
    return {"bf16": 2, "fp32": 4, "e4m3": 1}[dtype]


def _values(case, seed):
    """The tensors that a user's program has: a dict of CUDA tensors and factors."""
    gen = torch.Generator(device=DEVICE).manual_seed(int(seed))
    kind, D, hq, hkv = case["kind"], case["head_dim"], case["hq"], case["hkv"]
    dt = torch.float32 if case["dtype"] == "fp32" else torch.bfloat16

    def normal(*shape, std=1.0):
        return (torch.randn(shape, generator=gen, device=DEVICE, dtype=torch.bfloat16 if dt != torch.float32 else dt)
                * std).to(dt)

    x = {}
    if kind in ("train", "forward"):
        T = case["tokens"]
        x.update(q=normal(T, hq, D), k=normal(T, hkv, D), v=normal(T, hkv, D))
        if kind == "train":
            x["do"] = normal(T, hq, D)
        rows = T
    else:
        B, n = case["batch"], case["new"]
        lens = _cache_lens(case)
        rows = int(lens.max()) + n
        if case["paged"]:
            pages = [-(-(int(c) + n) // PAGE) for c in lens]
            order = np.random.Generator(np.random.PCG64(case["layout"] + 1)).permutation(sum(pages))
            table = np.zeros((B, max(pages)), np.int32)
            at = 0
            for b, m in enumerate(pages):
                table[b, :m] = order[at:at + m]
                at += m
            x["table_host"], x["table"] = table, torch.from_numpy(table.copy()).to(DEVICE)
            shape = (sum(pages) * PAGE, hkv, D)
        else:
            shape = (B, rows, hkv, D)
        x.update(k_cache=normal(*shape), v_cache=normal(*shape))
        # one call of n tokens, or n calls of one
        lead = (1, B, n) if kind == "append" else (n, B, 1)
        x.update(q=normal(*lead, hq, D), k=normal(*lead, hkv, D), v=normal(*lead, hkv, D))
        x["len_host"], x["len0"] = lens.copy(), torch.from_numpy(lens.copy()).to(DEVICE)
    if case["dtype"] == "e4m3":  # one factor per tensor, a cache and its new rows share it
        for name, parts in (("q", ["q"]), ("k", ["k", "k_cache"]), ("v", ["v", "v_cache"])):
            parts = [p for p in parts if p in x]
            top = max(float(x[p].float().abs().max()) for p in parts)
            x[name + "_factor"] = top / 448.0
            for p in parts:
                x[p] = (x[p].float() / x[name + "_factor"]).to(torch.float8_e4m3fn)
    if case["rope"]:
        x["cos"], x["sin"] = (torch.from_numpy(t).to(DEVICE) for t in wl.rope_tables(rows, D))
    return x


def prepare(case, seed):
    x = _values(case, seed)
    s = {"case": case, "x": x, "scale": case["head_dim"] ** -0.5}
    if case["kind"] in ("train", "forward"):
        s["segs"] = ism.Segments.from_workload(_segments(case), DEVICE)
        if case["plan"] != "none":
            s["plan"] = ism.Plan(s["segs"], case["hq"], case["hkv"], case["head_dim"], x["q"].dtype, DEVICE)
        return s
    n, B, hq, D = case["new"], case["batch"], case["hq"], case["head_dim"]
    s["end"] = [n] if case["kind"] == "append" else [1]
    s["type"] = [wl.QUERY if case["kind"] == "append" and case["query"] else wl.ANSWER]
    s["len"], s["host"] = x["len0"].clone(), x["len_host"].copy()
    lead = x["q"].shape
    s["o"] = torch.empty(lead, dtype=torch.bfloat16, device=DEVICE)
    s["lse"] = torch.empty((lead[0], hq, B, lead[2]), dtype=torch.float32, device=DEVICE)
    s["calls"] = [_append_call(case, s, i) for i in range(lead[0])]
    return s


def _append_call(case, s, i):
    """The i-th call of a pass, on its own new tokens and output rows."""
    x, scale = s["x"], s["scale"]
    q, k, v, o, lse = x["q"][i], x["k"][i], x["v"][i], s["o"][i], s["lse"][i]
    new = (q, k, v, x["k_cache"], x["v_cache"])
    lens = (s["len"], s["host"])
    segs = (s["end"], s["type"])
    if case["paged"]:
        table = (PAGE, x["table"], x["table_host"])
        if case["rope"]:
            return lambda: ism.prefill_append_paged_rope(*new, *table, *lens, *segs, x["cos"], x["sin"], scale,
                                                         out=o, lse=lse)
        return lambda: ism.prefill_append_paged(*new, *table, *lens, *segs, scale, out=o, lse=lse)
    if case["dtype"] == "e4m3":
        f = (x["q_factor"], x["k_factor"], x["v_factor"])
        return lambda: ism.prefill_append_e4m3(*new, *lens, *segs, *f, scale, out=o, lse=lse)
    rope = (x["cos"], x["sin"]) if case["rope"] else None
    if case["kind"] == "decode":  # a generation loop prepares its call
        return ism.AppendStep(*new, *lens, *segs, scale, out=o, lse=lse, rope=rope)
    if rope:
        return lambda: ism.prefill_append_rope(*new, *lens, *segs, *rope, scale, out=o, lse=lse)
    return lambda: ism.prefill_append(*new, *lens, *segs, scale, out=o, lse=lse)


def run(state):
    case, x, scale = state["case"], state["x"], state["scale"]
    if case["kind"] == "forward":
        o, lse = ism.fwd_e4m3(state["segs"], x["q"], x["k"], x["v"], x["q_factor"], x["k_factor"], x["v_factor"],
                              scale)
        return {"o": o, "lse": lse}
    if case["kind"] == "train":
        segs, plan = state["segs"], state.get("plan")
        if case["plan"] == "step":
            plan.build()
        low = case["min_workspace"]
        if case["rope"]:
            t = (x["cos"], x["sin"])
            o, lse, q, k = ism.fwd_rope(segs, x["q"], x["k"], x["v"], *t, scale, plan=plan)
            dq, dk, dv = ism.bwd_rope(segs, q, k, x["v"], o, lse, x["do"], *t, scale, minimal_workspace=low, plan=plan)
            return {"o": o, "lse": lse, "dq": dq, "dk": dk, "dv": dv, "q_rot": q, "k_rot": k}
        o, lse = ism.fwd(segs, x["q"], x["k"], x["v"], scale, plan=plan)
        dq, dk, dv = ism.bwd(segs, x["q"], x["k"], x["v"], o, lse, x["do"], scale, minimal_workspace=low, plan=plan)
        return {"o": o, "lse": lse, "dq": dq, "dk": dk, "dv": dv}
    # back to the dialogues as they stood before this turn (an answer given anew)
    state["len"].copy_(x["len0"])
    state["host"][:] = x["len_host"]
    for call in state["calls"]:
        call()
        state["host"] += case["new"] if case["kind"] == "append" else 1
    return {"o": state["o"], "lse": state["lse"], "k_cache": x["k_cache"], "v_cache": x["v_cache"],
            "len": state["len"]}


# ----------------------------------------------------------- work and accuracy

def work(case):
    """Contractions over the visible pairs (forward Q K^T and P V; backward Q K^T, dO V^T, dV, dK and dQ), every
    input read once and every output written once."""
    D, hq, hkv, kind = case["head_dim"], case["hq"], case["hkv"], case["kind"]
    pairs, e = _visible(case) * hq, _bytes_of(case["dtype"])
    if kind == "train":
        T = case["tokens"]
        rows = 5 * hq + 6 * hkv + (2 * (hq + hkv) if case["rope"] else 0)  # q, o, do, o, dq and k, v, k, v, dk, dv
        return {"bytes": T * D * e * rows + 4 * T * hq * 2, "flops": 14 * D * pairs}
    if kind == "forward":
        T = case["tokens"]
        return {"bytes": T * D * (hq + 2 * hkv) * e + T * hq * (2 * D + 4), "flops": 4 * D * pairs}
    B, n = case["batch"], case["new"]
    reads = 1 if kind == "append" else n  # a decode reads the cache for each token
    cached = int(_cache_lens(case).sum()) * reads * 2 * hkv * D * e
    new = B * n * (D * (hq + 4 * hkv) * e + hq * (2 * D + 4))
    return {"bytes": cached + new, "flops": 4 * D * pairs}


def tolerance(case):
    if case["dtype"] == "fp32":
        return {"rel": 1e-5}
    if case["dtype"] == "e4m3":
        return {"rel": 0.03}
    return {"rel": 1e-2}


def _rotate(x, cos, sin):
    """Rotate-half rotary encoding of x [L, H, D] in 64 bits."""
    h = x.shape[-1] // 2
    a, b = x[..., :h], x[..., h:]
    c, s = cos[:, None, :], sin[:, None, :]
    return torch.cat([a * c - b * s, b * c + a * s], dim=-1)


def _attend(q, k, v, ends, scale, do=None):
    """One dialogue in 64 bits: q [L, Hq, D], k / v [K, Hkv, D], ends [L]; (o, lse) or, with do, the gradients too."""
    L, hq, D = q.shape
    group = hq // k.shape[1]
    o, lse = torch.empty_like(q), q.new_empty((hq, L))
    dq, dk, dv = torch.zeros_like(q), torch.zeros_like(k), torch.zeros_like(v)
    for r0 in range(0, L, 2048):
        r1 = min(L, r0 + 2048)
        m = int(ends[r0:r1].max())
        hidden = torch.arange(m, device=q.device)[None, :] >= ends[r0:r1, None]
        for h in range(hq):
            qh, kh, vh = q[r0:r1, h], k[:m, h // group], v[:m, h // group]
            s = (qh @ kh.T).mul_(scale).masked_fill_(hidden, -math.inf)
            z = torch.logsumexp(s, dim=1)
            p = s.sub_(z[:, None]).exp_()
            o[r0:r1, h], lse[h, r0:r1] = p @ vh, z
            if do is not None:
                g = do[r0:r1, h]
                dv[:m, h // group] += p.T @ g
                ds = (g @ vh.T).sub_((g * o[r0:r1, h]).sum(1, keepdim=True)).mul_(p).mul_(scale)
                dq[r0:r1, h] = ds @ kh
                dk[:m, h // group] += ds.T @ qh
    return (o, lse) if do is None else (o, lse, dq, dk, dv)


def exact(case, seed):
    """What run() returns, in 64 bits; None for the copied caches."""
    if work(case)["flops"] > 8e12:  # about 10 s in 64 bits
        return None
    x, scale, kind = _values(case, seed), case["head_dim"] ** -0.5, case["kind"]

    def f64(name):
        return x[name].to(torch.float64) * x.get(name.split("_")[0] + "_factor", 1.0)

    if kind in ("train", "forward"):
        segs = _segments(case)
        q, k, v = f64("q"), f64("k"), f64("v")
        do = f64("do") if kind == "train" else None
        parts = []
        for b in range(segs.num_seqs):
            t0, L, se, st = segs.seq(b)
            rows = slice(t0, t0 + L)
            qb, kb = q[rows], k[rows]
            if case["rope"]:
                c, s = x["cos"][:L].double(), x["sin"][:L].double()
                qb, kb = _rotate(qb, c, s), _rotate(kb, c, s)
            got = list(_attend(qb, kb, v[rows], torch.from_numpy(_ends(se, st)).to(DEVICE), scale,
                               None if do is None else do[rows]))
            if case["rope"]:
                got[2:4] = [_rotate(g, c, -s) for g in got[2:4]]
                got += [qb, kb]
            parts.append(got)
        names = ["o", "lse", "dq", "dk", "dv", "q_rot", "k_rot"]
        return {n: torch.cat(p, dim=1 if n == "lse" else 0) for n, p in zip(names, zip(*parts))}
    n, B = case["new"], case["batch"]
    qs, ks, vs = f64("q"), f64("k"), f64("v")
    o = torch.empty(qs.shape, dtype=torch.float64, device=DEVICE)
    lse = torch.empty((qs.shape[0], case["hq"], B, qs.shape[2]), dtype=torch.float64, device=DEVICE)
    for b in range(B):
        c = int(x["len_host"][b])
        if case["paged"]:
            at = np.arange(c)
            at = torch.from_numpy(x["table_host"][b, at // PAGE].astype(np.int64) * PAGE + at % PAGE).to(DEVICE)
            hist = [x[w][at] for w in ("k_cache", "v_cache")]
        else:
            hist = [x[w][b, :c] for w in ("k_cache", "v_cache")]
        k, v = (h.to(torch.float64) * x.get(w, 1.0) for h, w in zip(hist, ("k_factor", "v_factor")))
        # the pass's n new tokens of this sequence, one call after the other
        qn, kn, vn = (t[:, b].flatten(0, 1) for t in (qs, ks, vs))
        if case["rope"]:
            t = [x[w][c:c + n].double() for w in ("cos", "sin")]
            qn, kn = _rotate(qn, *t), _rotate(kn, *t)
        ends = torch.full((n,), c + n, device=DEVICE) if kind == "append" and case["query"] else \
            torch.arange(c + 1, c + n + 1, device=DEVICE)
        ob, lb = _attend(qn, torch.cat([k, kn]), torch.cat([v, vn]), ends, scale)
        if kind == "append":
            o[0, b], lse[0, :, b] = ob, lb
        else:
            o[:, b, 0], lse[:, :, b, 0] = ob, lb.T
    return {"o": o, "lse": lse, "k_cache": None, "v_cache": None, "len": None}
