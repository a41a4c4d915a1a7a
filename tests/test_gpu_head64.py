"""bf16 at head_dim 64 on the tensor cores: forward, backward, rotary pair,
plans and appends against the fp64 oracle, at tile edges and remainders.

Tolerance: P and dS carry 16 mantissa bits into their contractions and every
sum is fp32, so a result is the exact one up to about 2^-16 relative plus the
bf16 output rounding, at most 2^-9 of each element: the 2-norm of the error is
at most (2^-9 + 2^-14) of the result's (2^-14 for the inner roundings and the
fp32 sums of up to a few hundred terms).  bf16 P or dS would give 2.2e-3 to
2.9e-3 and fail.
"""
import numpy as np
import pytest
import torch

from oracle import ism_oracle as orc
from paper_2408_00539_gb300 import ism
from paper_2408_00539_gb300 import workloads as wl

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
REL = 2.0 ** -9 + 2.0 ** -14
D = 64

# lengths around one and two tiles, several tiles with a remainder, one token
DIALOGUES = [([1], [1]), ([40, 127], [0, 1]), ([128], [0]), ([60, 129], [1, 0]),
             ([70, 150, 170, 300, 385], [0, 1, 0, 1, 0]), ([0, 64, 64, 256], [1, 0, 1, 1])]


def _rel(got, ref):
    got, ref = got.double().cpu().numpy(), np.asarray(ref, dtype=np.float64)
    assert np.isfinite(got).all()
    return np.linalg.norm(got - ref) / np.linalg.norm(ref)


def _inputs(hq, hkv, seed=11):
    w = wl.Workload("d64", wl.pack(DIALOGUES), hq, hkv, D, "bf16", D ** -0.5, 1.0, seed)
    return w, wl.attention_tensors(w)


@pytest.mark.parametrize("hq,hkv", [(1, 1), (4, 2), (6, 2), (3, 3), (8, 1)])
def test_forward_backward(hq, hkv):
    w, (q, k, v, do) = _inputs(hq, hkv)
    segs = ism.Segments.from_workload(w.segs, DEV)
    qd, kd, vd, dod = (t.to(DEV) for t in (q, k, v, do))
    o, lse = ism.fwd(segs, qd, kd, vd, w.softmax_scale)
    grads = ism.bwd(segs, qd, kd, vd, o, lse, dod, w.softmax_scale)
    ism.check_status(DEV)
    o_ref, lse_ref = orc.attn_fwd(q, k, v, w.segs, w.softmax_scale)
    assert _rel(o, o_ref) <= REL
    assert np.abs(lse.cpu().numpy() - lse_ref).max() <= 1e-5
    # the backward's Delta comes from the bf16 O (2^-9 of it), which the
    # oracle's does not: compared on the rounded O
    for got, ref in zip(grads, orc.attn_bwd(q, k, v, do, w.segs, w.softmax_scale)):
        assert _rel(got, ref) <= REL + 2.0 ** -12
    # a plan of the same heads, whatever element type it was built for
    for dt in (torch.bfloat16, torch.float32):
        plan = ism.Plan(segs, hq, hkv, D, dt, DEV)
        o2, lse2 = ism.fwd(segs, qd, kd, vd, w.softmax_scale, plan=plan)
        g2 = ism.bwd(segs, qd, kd, vd, o, lse, dod, w.softmax_scale, plan=plan)
        for a, b in zip((o2, lse2, *g2), (o, lse, *grads)):
            assert torch.equal(a, b)


@pytest.mark.parametrize("hq,hkv", [(2, 2), (3, 1), (4, 1)])
def test_rotary(hq, hkv):
    w, (q, k, v, do) = _inputs(hq, hkv, 12)
    segs = ism.Segments.from_workload(w.segs, DEV)
    cos, sin = (torch.from_numpy(t) for t in wl.rope_tables(400, D))
    qd, kd, vd, dod, cd, sd = (t.to(DEV) for t in (q, k, v, do, cos, sin))
    o, lse, qr, kr = ism.fwd_rope(segs, qd, kd, vd, cd, sd, w.softmax_scale)
    dq, dk, dv = ism.bwd_rope(segs, qr, kr, vd, o, lse, dod, cd, sd, w.softmax_scale)
    ism.check_status(DEV)
    # gradients of the rotated rows, turned back by the opposite angles
    rq, rk, rv = orc.attn_bwd(qr.cpu(), kr.cpu(), v, do, w.segs, w.softmax_scale)
    pos = np.concatenate([np.arange(e[-1]) for e, _ in DIALOGUES])
    c, s = (t.double().numpy()[pos][:, None, :] for t in (cos, sin))
    h = D // 2
    for got, g in ((dq, rq), (dk, rk)):
        ref = np.concatenate([g[..., :h] * c + g[..., h:] * s, g[..., h:] * c - g[..., :h] * s], -1)
        assert _rel(got, ref) <= REL + 2.0 ** -12
    assert _rel(dv, rv) <= REL
    assert _rel(o, orc.attn_fwd(qr.cpu(), kr.cpu(), v, w.segs, w.softmax_scale)[0]) <= REL


@pytest.mark.parametrize("hq,hkv,ln", [(4, 2, 2), (3, 1, 130), (8, 2, 257)])
def test_append(hq, hkv, ln):
    """A chunk against caches whose rows past the lengths hold NaN."""
    lens, cap = np.array([1, 127, 300], np.int32), 600
    gen = torch.Generator().manual_seed(5)
    B = len(lens)
    q, k, v = (torch.randn((B, ln, h, D), generator=gen).bfloat16() for h in (hq, hkv, hkv))
    kc, vc = (torch.randn((B, cap, hkv, D), generator=gen).bfloat16() for _ in range(2))
    kd, vd = kc.to(DEV), vc.to(DEV)
    for b, c in enumerate(lens):
        kd[b, c:], vd[b, c:] = float("nan"), float("nan")
    ends, types = [ln // 2, ln], [0, 1]
    o, _ = ism.prefill_append(q.to(DEV), k.to(DEV), v.to(DEV), kd, vd, torch.from_numpy(lens.copy()).to(DEV), lens,
                              ends, types, D ** -0.5)
    ism.check_status(DEV)
    for b, c in enumerate(lens):
        whole = wl.pack([([int(c)] + [int(c) + e for e in ends], [1] + types)])
        full = [torch.cat([x[b, :c], n[b]]) for x, n in ((kc, k), (vc, v))]
        qf = torch.cat([torch.zeros((int(c), hq, D), dtype=torch.bfloat16), q[b]])
        ref = orc.attn_fwd(qf, *full, whole, D ** -0.5)[0][c:]
        assert _rel(o[b], ref) <= REL


def _cuda_cores(monkeypatch, call):
    monkeypatch.setenv("ISM_FORCE_CUDA_CORES", "1")
    ism.load().ism_debug_reload_env()
    try:
        return call()
    finally:
        monkeypatch.delenv("ISM_FORCE_CUDA_CORES")
        ism.load().ism_debug_reload_env()


def _same_reach(got, ref, rel=2 * REL):
    """NaN and Inf in the same places, and the finite values those of the
    reference to within both roundings."""
    a, b = (t.double().cpu().numpy() for t in (got, ref))
    assert np.array_equal(np.isnan(a), np.isnan(b))
    inf = np.isinf(a)
    assert np.array_equal(inf, np.isinf(b)) and np.array_equal(a[inf], b[inf])
    ok = np.isfinite(a)
    assert np.linalg.norm(a[ok] - b[ok]) <= rel * np.linalg.norm(b[ok])
    return ok.mean()


BAD = [("q", "nan"), ("k", "nan"), ("v", "nan"), ("do", "nan"), ("v", "inf"), ("do", "inf"), ("k", "-inf")]


@pytest.mark.parametrize("name,value", BAD)
@pytest.mark.parametrize("hq,hkv,rope", [(4, 2, False), (3, 1, False), (4, 2, True)])
def test_reach_of_nan_and_inf(monkeypatch, name, value, hq, hkv, rope):
    """A NaN or Inf in one row reaches what the mask lets it reach and nothing
    beside it, neither in its own dialogue nor in its neighbours'.  Reference:
    the CUDA-core kernels, which read visible rows only."""
    w = wl.Workload("d64", wl.pack([([50], [1]), ([30, 400], [0, 1]), ([50], [0]), ([260], [1])]), hq, hkv, D, "bf16",
                    D ** -0.5, 1.0, 14)
    x = dict(zip(("q", "k", "v", "do"), wl.attention_tensors(w)))
    x[name][50 + 150, 0] = float(value)
    segs = ism.Segments.from_workload(w.segs, DEV)
    q, k, v, do = (t.to(DEV) for t in x.values())
    tables = tuple(torch.from_numpy(t).to(DEV) for t in wl.rope_tables(500, D))

    def step():
        if rope:
            o, lse, qr, kr = ism.fwd_rope(segs, q, k, v, *tables, w.softmax_scale)
            out = (o, lse, *ism.bwd_rope(segs, qr, kr, v, o, lse, do, *tables, w.softmax_scale))
        else:
            o, lse = ism.fwd(segs, q, k, v, w.softmax_scale)
            out = (o, lse, *ism.bwd(segs, q, k, v, o, lse, do, w.softmax_scale))
        ism.check_status(DEV)
        return out

    got, ref = step(), _cuda_cores(monkeypatch, step)
    finite = [_same_reach(a, b, 1e-5 if i == 1 else 2 * REL) for i, (a, b) in enumerate(zip(got, ref))]
    assert 0.4 < min(finite) < 1.0


@pytest.mark.parametrize("hq,hkv,cached", [(4, 2, 3000), (4, 2, 10), (3, 1, 1000)])
@pytest.mark.parametrize("value", ["nan", "inf"])
def test_reach_in_an_append(monkeypatch, hq, hkv, cached, value):
    """A bad value row among the new ones: earlier rows of the chunk do not see it."""
    ln, lens = 150, np.array([cached], np.int32)
    gen = torch.Generator().manual_seed(7)
    new = [torch.randn((1, ln, h, D), generator=gen).bfloat16() for h in (hq, hkv, hkv)]
    caches = [torch.randn((1, cached + ln, hkv, D), generator=gen).bfloat16() for _ in range(2)]
    new[2][0, 60, 0] = float(value)

    def call():
        o, lse = ism.prefill_append(*(t.to(DEV) for t in new + caches), torch.from_numpy(lens.copy()).to(DEV), lens,
                                    [ln], [1], D ** -0.5)
        ism.check_status(DEV)
        return o, lse

    got, ref = call(), _cuda_cores(monkeypatch, call)
    assert 0.3 < _same_reach(got[0], ref[0]) < 1.0
    assert _same_reach(got[1], ref[1], 1e-5) == 1.0
