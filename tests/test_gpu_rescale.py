"""The lazy rescale of the running maximum where only some rows of a warp need
it: scores of a wide spread (standard deviation 5 before the softmax), so that
the maximum of a later key tile exceeds an earlier one by more than 2^8 in some
rows and not in others.  The reference is the fp64 oracle.

Tolerance in the 2-norm: P is rounded to bf16 (2^-9 of its term; to e4m3, 2^-4)
and the output to bf16 (2^-9), and the fp32 scores of size up to 25 carry 2^-24
each of it: 2 * 2^-9 + 2^-14, or 4e-2 for e4m3 (uniform roundings of zero mean).
"""
import numpy as np
import pytest
import torch

from oracle import ism_oracle as orc
from paper_2408_00539_gb300 import ism
from paper_2408_00539_gb300 import workloads as wl

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
DIALOGUES = [([70, 150, 170, 300, 700], [0, 1, 0, 1, 0]), ([129], [0]), ([60, 257, 400], [1, 0, 1])]
REL = 2 * 2.0 ** -9 + 2.0 ** -14
SPREAD = 5.0 ** 0.5  # of q and of k each


def _inputs(hq, hkv, d):
    w = wl.Workload("spread", wl.pack(DIALOGUES), hq, hkv, d, "bf16", d ** -0.5, 1.0, 17)
    q, k, v, do = wl.attention_tensors(w)
    return w, [(q * SPREAD).bfloat16(), (k * SPREAD).bfloat16(), v, do]


def _some_rows_rescale(q, k, segs, scale):
    """Whether the rows of some warp (32 in a row of head 0, the last query of
    the longest dialogue) differ in needing a rescale."""
    t0, n, _, _ = segs.seq(0)
    s = q[t0 + 320:t0 + 672, 0].float() @ k[t0:t0 + n, 0].float().T * scale * 1.4427
    need = (s[:, 128:256].max(1).values > s[:, :128].max(1).values + 8).view(-1, 32)
    return bool((need.any(1) & ~need.all(1)).any())


def _rel(got, ref):
    got = got.double().cpu().numpy()
    assert np.isfinite(got).all()
    return np.linalg.norm(got - ref) / np.linalg.norm(ref)


@pytest.mark.parametrize("hq,hkv,d,one_head", [(8, 2, 128, False), (3, 3, 128, False), (4, 2, 64, False),
                                               (3, 1, 64, False), (3, 3, 128, True)])
def test_forward_backward(monkeypatch, hq, hkv, d, one_head):
    w, x = _inputs(hq, hkv, d)
    assert _some_rows_rescale(x[0], x[1], w.segs, w.softmax_scale)
    if one_head:
        monkeypatch.setenv("ISM_FWD_ONE_HEAD", "1")
    ism.load().ism_debug_reload_env()
    try:
        segs = ism.Segments.from_workload(w.segs, DEV)
        dev = [t.to(DEV) for t in x]
        o, lse = ism.fwd(segs, *dev[:3], w.softmax_scale)
        grads = ism.bwd(segs, *dev[:3], o, lse, dev[3], w.softmax_scale)
        ism.check_status(DEV)
    finally:
        monkeypatch.delenv("ISM_FWD_ONE_HEAD", raising=False)
        ism.load().ism_debug_reload_env()
    ref, lse_ref = orc.attn_fwd(*x[:3], w.segs, w.softmax_scale)
    assert _rel(o, ref) <= REL
    assert np.abs(lse.cpu().numpy() - lse_ref).max() <= 1e-4
    for a, b in zip(grads, orc.attn_bwd(*x, w.segs, w.softmax_scale)):
        assert _rel(a, b) <= 3 * 2.0 ** -9  # (P, dS and the output; Delta from the bf16 O)


@pytest.mark.parametrize("hq,hkv", [(4, 2), (3, 1)])
def test_e4m3(hq, hkv):
    w, x = _inputs(hq, hkv, 128)
    factor = [float(t.float().abs().max()) / 448 for t in x[:3]]
    e8 = [(t.float() / f).to(torch.float8_e4m3fn) for t, f in zip(x, factor)]
    o, _ = ism.fwd_e4m3(ism.Segments.from_workload(w.segs, DEV), *(t.to(DEV) for t in e8), *factor, w.softmax_scale)
    ism.check_status(DEV)
    exact = [t.double() * f for t, f in zip(e8, factor)]
    assert _rel(o, orc.attn_fwd(*exact, w.segs, w.softmax_scale)[0]) <= 4e-2


@pytest.mark.parametrize("hq,hkv,d,ln", [(8, 2, 128, 40), (4, 2, 64, 40), (3, 3, 128, 40), (3, 3, 128, 200)])
def test_append(hq, hkv, d, ln):
    """Against a cache, split over its keys and not (a whole item's tiles follow one another)."""
    gen = torch.Generator().manual_seed(6)
    c, cap = 1000, 1300
    q, k, v, kc, vc = ((torch.randn((1, n, h, d), generator=gen) * f).bfloat16() for n, h, f in (
        (ln, hq, SPREAD), (ln, hkv, SPREAD), (ln, hkv, 1.0), (cap, hkv, SPREAD), (cap, hkv, 1.0)))
    lens = np.array([c], np.int32)
    o, _ = ism.prefill_append(*(t.to(DEV) for t in (q, k, v, kc, vc)), torch.from_numpy(lens.copy()).to(DEV), lens,
                              [ln], [0], d ** -0.5)
    ism.check_status(DEV)
    whole = [torch.cat([a[0, :c], b[0]]) for a, b in ((kc, k), (vc, v))]
    qf = torch.cat([torch.zeros((c, hq, d), dtype=torch.bfloat16), q[0]])
    ref = orc.attn_fwd(qf, *whole, wl.pack([([c, c + ln], [1, 0])]), d ** -0.5)[0][c:]
    assert _rel(o[0], ref) <= REL
