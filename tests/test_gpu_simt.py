"""The CUDA-core kernels (fp32; bf16 under ISM_FORCE_CUDA_CORES=1) at the edges
of their blocks: 16- and 64-row blocks, head_dim 64 and 128, odd groups,
remainders, one token, and rows holding NaN that others do not see.

Tolerance of the fp32 results: every sum is fp32 over at most a few hundred
terms, 2^-24 each, and expf adds 2 ulp; 1e-5 is over ten times that.
"""
import numpy as np
import pytest
import torch

from oracle import ism_oracle as orc
from paper_2408_00539_gb300 import ism
from paper_2408_00539_gb300 import workloads as wl

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
DIALOGUES = [([1], [1]), ([15], [0]), ([10, 17], [1, 0]), ([40, 63], [0, 1]), ([65], [1]), ([60, 129], [0, 1]),
             ([70, 150, 170, 300], [0, 1, 0, 1])]


def _rel(got, ref):
    return np.linalg.norm(got.double().cpu().numpy() - ref) / np.linalg.norm(ref)


def _run(segs, q, k, v, do, scale):
    s = ism.Segments.from_workload(segs, DEV)
    q, k, v, do = (t.to(DEV) for t in (q, k, v, do))
    o, lse = ism.fwd(s, q, k, v, scale)
    out = (o, lse, *ism.bwd(s, q, k, v, o, lse, do, scale))
    ism.check_status(DEV)
    return out


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("hq,hkv,copies", [(1, 1, 1), (6, 2, 1), (4, 4, 12)])  # the last one: blocks of 64 rows
def test_fp32(d, hq, hkv, copies):
    w = wl.Workload("simt", wl.pack(DIALOGUES * copies), hq, hkv, d, "fp32", d ** -0.5, 1.0, 3)
    q, k, v, do = wl.attention_tensors(w)
    got = _run(w.segs, q, k, v, do, w.softmax_scale)
    ref = (*orc.attn_fwd(q, k, v, w.segs, w.softmax_scale), *orc.attn_bwd(q, k, v, do, w.segs, w.softmax_scale))
    for a, b in zip(got, ref):
        assert _rel(a, b) <= 1e-5


@pytest.mark.parametrize("d", [64, 128])
def test_unseen_nan(d):
    """A NaN answer token (K, V, Q, dO) reaches no earlier row's output and no
    gradient of a key that only earlier rows see."""
    segs = wl.pack([([30, 200], [0, 1]), ([50], [0])])
    w = wl.Workload("nan", segs, 2, 1, d, "fp32", d ** -0.5, 1.0, 4)
    x = wl.attention_tensors(w)
    clean = _run(segs, *x, w.softmax_scale)
    at = 150
    for t in x[:3]:
        t[at] = float("nan")
    o, lse, dq, dk, dv = _run(segs, *x, w.softmax_scale)
    for a, b in ((o, clean[0]), (dq, clean[2])):
        assert torch.equal(a[:at], b[:at]) and torch.equal(a[200:], b[200:])
    assert torch.equal(lse[:, :at], clean[1][:, :at])
    for a, b in ((dk, clean[3]), (dv, clean[4])):
        assert torch.equal(a[200:], b[200:])
        assert torch.isnan(a[at]).all()


@pytest.mark.parametrize("d", [64, 128])
def test_bf16_forced(d, monkeypatch):
    w = wl.Workload("simt16", wl.pack(DIALOGUES), 3, 1, d, "bf16", d ** -0.5, 1.0, 6)
    x = wl.attention_tensors(w)
    monkeypatch.setenv("ISM_FORCE_CUDA_CORES", "1")
    ism.load().ism_debug_reload_env()
    try:
        got = _run(w.segs, *x, w.softmax_scale)
    finally:
        monkeypatch.delenv("ISM_FORCE_CUDA_CORES")
        ism.load().ism_debug_reload_env()
    ref = (*orc.attn_fwd(*x[:3], w.segs, w.softmax_scale), *orc.attn_bwd(*x, w.segs, w.softmax_scale))
    for a, b in zip(got, ref):  # the bf16 output rounding (and Delta from the bf16 O)
        assert _rel(a, b) <= 2.0 ** -9 + 2.0 ** -12


@pytest.mark.parametrize("hq,hkv,d", [(3, 1, 64), (3, 3, 128), (4, 2, 64)])
@pytest.mark.parametrize("copies", [2, 40])  # the small metadata pass and the general one
def test_query_tiles_in_cost_order(hq, hkv, d, copies):
    """The fp32 forward takes the most expensive query tiles first, whatever the
    group; a plan of an odd group has the even-indexed tiles in front and each
    half in order, and gives the same results."""
    segs = wl.pack([([70, 150, 170, 700], [0, 1, 0, 1]), ([129], [0]), ([400], [1]), ([1], [1])] * copies)
    w = wl.Workload("order", segs, hq, hkv, d, "fp32", d ** -0.5, 1.0, 8)
    q, k, v, do = (t.to(DEV) for t in wl.attention_tensors(w))
    s = ism.Segments.from_workload(segs, DEV)
    T, nq = w.total_tokens, sum(-(-segs.seq(b)[1] // 128) for b in range(segs.num_seqs))
    up = lambda n: (n + 255) // 256 * 256

    def lists(buffer):  # (tile index in its dialogue, key tiles) along q_order
        words = buffer.cpu().numpy().view(np.int32)
        tiles = words[up(4 * T) // 4:][:8 * nq].reshape(nq, 8)
        order = words[(up(4 * T) + up(32 * nq)) // 4:][:nq]
        assert sorted(order) == list(range(nq))
        return tiles[order, 4], tiles[order, 6]

    ws = ism._workspace(64 << 20, DEV)
    o, lse = ism.fwd(s, q, k, v, w.softmax_scale, workspace=ws)
    grads = ism.bwd(s, q, k, v, o, lse, do, w.softmax_scale)
    cost = lists(ws)[1]
    assert (np.diff(cost) <= 0).all()
    plan = ism.Plan(s, hq, hkv, d, torch.float32, DEV)
    index, cost = lists(plan.buffer)
    if (hq // hkv) % 2:
        heads = int((index % 2 == 0).sum())
        assert (index[:heads] % 2 == 0).all() and (np.diff(cost[heads:]) <= 0).all()
    else:
        assert (np.diff(cost) <= 0).all()
    o2, lse2 = ism.fwd(s, q, k, v, w.softmax_scale, plan=plan)
    for a, b in zip((o, lse, *grads), (o2, lse2, *ism.bwd(s, q, k, v, o, lse, do, w.softmax_scale, plan=plan))):
        assert torch.equal(a, b)
    ism.check_status(DEV)
