"""Kernels launched as programmatic dependents: the same results under stream
capture (several replays), back to back without a synchronisation, on inputs
written by the kernel just before, and on two streams at once.  Also the small
metadata pass against the tile map's own arrays."""
import numpy as np
import pytest
import torch

from paper_2408_00539_gb300 import ism
from paper_2408_00539_gb300 import workloads as wl

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
DIALOGUES = [([70, 150, 170, 300], [0, 1, 0, 1]), ([129], [0]), ([1], [1]), ([60, 257, 400], [1, 0, 1])]


def _step(segs, x, scale, plan=None, rope=None):
    if rope is None:
        o, lse = ism.fwd(segs, *x[:3], scale, plan=plan)
        return (o, lse, *ism.bwd(segs, *x[:3], o, lse, x[3], scale, plan=plan))
    o, lse, q, k = ism.fwd_rope(segs, *x[:3], *rope, scale, plan=plan)
    return (o, lse, *ism.bwd_rope(segs, q, k, x[2], o, lse, x[3], *rope, scale, plan=plan))


@pytest.mark.parametrize("hq,hkv,d,dtype", [(8, 2, 128, "bf16"), (3, 1, 128, "bf16"), (4, 2, 64, "bf16"),
                                            (2, 2, 64, "fp32")])
@pytest.mark.parametrize("planned", [False, True])
@pytest.mark.parametrize("rope", [False, True])
def test_training_step(hq, hkv, d, dtype, planned, rope):
    w = wl.Workload("pdl", wl.pack(DIALOGUES), hq, hkv, d, dtype, d ** -0.5, 1.0, 31)
    host = [t for t in wl.attention_tensors(w)]
    segs = ism.Segments.from_workload(w.segs, DEV)
    x = [t.to(DEV) for t in host]
    tables = tuple(torch.from_numpy(t).to(DEV) for t in wl.rope_tables(500, d)) if rope else None
    plan = ism.Plan(segs, hq, hkv, d, x[0].dtype, DEV) if planned else None
    torch.cuda.synchronize()
    ref = [t.clone() for t in _step(segs, x, w.softmax_scale, plan, tables)]
    ism.check_status(DEV)
    # inputs written by the kernel just before, many steps without a wait
    live = [torch.zeros_like(t) for t in x]
    outs = []
    for _ in range(6):
        for a, b in zip(live, x):
            torch.mul(b, 1.0, out=a)
        outs.append(_step(segs, live, w.softmax_scale, plan, tables))
        for a in live:
            a.zero_()
    ism.check_status(DEV)
    for out in outs:
        assert all(torch.equal(a, b) for a, b in zip(out, ref))
    # captured
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        out = _step(segs, x, w.softmax_scale, plan, tables)
    for _ in range(3):
        for t in out:
            t.zero_()
        g.replay()
        torch.cuda.synchronize()
        assert all(torch.equal(a, b) for a, b in zip(out, ref))


def test_two_streams():
    w = wl.Workload("pdl", wl.pack(DIALOGUES * 8), 8, 2, 128, "bf16", 128 ** -0.5, 1.0, 32)
    x = [t.to(DEV) for t in wl.attention_tensors(w)]
    segs = ism.Segments.from_workload(w.segs, DEV)
    ref = [t.clone() for t in _step(segs, x, w.softmax_scale)]
    streams = [torch.cuda.Stream(DEV) for _ in range(2)]
    outs = []
    torch.cuda.synchronize()
    for _ in range(4):
        for s in streams:
            with torch.cuda.stream(s):
                outs.append(_step(segs, x, w.softmax_scale))
    torch.cuda.synchronize()
    ism.check_status(DEV)
    for out in outs:
        assert all(torch.equal(a, b) for a, b in zip(out, ref))


@pytest.mark.parametrize("new", [1, 40])
@pytest.mark.parametrize("rope", [False, True])
def test_append_captured(new, rope):
    lens = np.array([300, 5, 128], np.int32)
    gen = torch.Generator().manual_seed(4)
    q, k, v = (torch.randn((3, new, h, 128), generator=gen).bfloat16().to(DEV) for h in (8, 2, 2))
    kc, vc = (torch.randn((3, 512, 2, 128), generator=gen).bfloat16().to(DEV) for _ in range(2))
    len0 = torch.from_numpy(lens.copy()).to(DEV)
    cl, o = len0.clone(), torch.empty_like(q)
    lse = torch.empty((8, 3, new), device=DEV)
    t = tuple(torch.from_numpy(a).to(DEV) for a in wl.rope_tables(600, 128)) if rope else None
    ws = ism._workspace(ism.append_workspace_size(q, k, 0.09, rope=rope), DEV)

    def call():
        cl.copy_(len0)
        args = (q, k, v, kc, vc, cl, lens, [new], [1])
        if rope:
            ism.prefill_append_rope(*args, *t, 0.09, out=o, lse=lse, workspace=ws)
        else:
            ism.prefill_append(*args, 0.09, out=o, lse=lse, workspace=ws)

    call()
    ism.check_status(DEV)
    ref = [x.clone() for x in (o, lse, kc, vc, cl)]
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        call()
    for _ in range(3):
        o.zero_()
        g.replay()
        torch.cuda.synchronize()
        assert all(torch.equal(a, b) for a, b in zip((o, lse, kc, vc, cl), ref))


@pytest.mark.parametrize("seed", range(6))
def test_small_and_general_metadata_agree(seed, monkeypatch):
    """The small pass serves up to 256 tiles and sequences and 1024 segments;
    the same dialogues beyond that go through the general one: the results of
    the leading dialogues must not change."""
    rng = np.random.default_rng(seed)
    few = wl.random_dialogue_set(rng, 12, 700)
    dialogues = [(few.seq(b)[2].tolist(), few.seq(b)[3].tolist()) for b in range(few.num_seqs)]
    many = wl.pack(dialogues + [([1], [1])] * 260)  # over 256 sequences
    w = wl.Workload("meta", many, 3, 1, 128, "bf16", 128 ** -0.5, 1.0, seed)
    x = [t.to(DEV) for t in wl.attention_tensors(w)]
    T = few.total_tokens
    a = _step(ism.Segments.from_workload(many, DEV), x, w.softmax_scale)
    b = _step(ism.Segments.from_workload(few, DEV), [t[:T].contiguous() for t in x], w.softmax_scale)
    ism.check_status(DEV)
    for name, y, z in zip("o lse dq dk dv".split(), a, b):
        assert torch.equal(y[:, :T] if name == "lse" else y[:T], z), name


def _decode_64(waits, paged, rope, stream):
    """64 steps of three caches on a stream; the new rows of each step are
    written into the same buffers by the kernel just before it."""
    lens = np.array([300, 5, 121], np.int32)  # every cache crosses into its next tile of 128 on the way
    gen = torch.Generator().manual_seed(8)
    B, n, hq, hkv = 3, 64, 8, 2
    new = [torch.randn((n, B, 1, h, 128), generator=gen).bfloat16().to(DEV) for h in (hq, hkv, hkv)]
    rows = (9 * 128, hkv, 128) if paged else (B, 400, hkv, 128)
    kc, vc = (torch.randn(rows, generator=gen).bfloat16().to(DEV) for _ in range(2))
    table = np.arange(9, dtype=np.int32)[::-1].reshape(3, 3).copy()
    dev_table, cl, host = torch.from_numpy(table).to(DEV), torch.from_numpy(lens.copy()).to(DEV), lens.copy()
    tables = tuple(torch.from_numpy(a).to(DEV) for a in wl.rope_tables(400, 128))
    x = [torch.empty_like(t[0]) for t in new]
    outs = []
    torch.cuda.synchronize()
    with torch.cuda.stream(stream):
        for i in range(n):
            for a, b in zip(x, new):
                torch.mul(b[i], 1.0, out=a)
            args = (cl, host, [1], [1])
            if paged:
                o = ism.prefill_append_paged(*x, kc, vc, 128, dev_table, table, *args, 0.09)
            elif rope:
                o = ism.prefill_append_rope(*x, kc, vc, *args, *tables, 0.09)
            else:
                o = ism.prefill_append(*x, kc, vc, *args, 0.09)
            outs.append(o)
            host += 1
            if waits:
                torch.cuda.synchronize()
    return outs, kc, vc, cl


@pytest.mark.parametrize("paged,rope", [(False, False), (True, False), (False, True)])
def test_decode_steps_back_to_back(paged, rope):
    """Steps without a wait, on two streams, against the same steps with a wait
    after each: the decode reads lengths, page table and old rows before the
    cache write in front of it is complete."""
    streams = [torch.cuda.Stream(DEV) for _ in range(2)]
    ref = _decode_64(True, paged, rope, streams[0])
    ism.check_status(DEV)
    got = [_decode_64(False, paged, rope, s) for s in streams for _ in range(2)]
    torch.cuda.synchronize()
    ism.check_status(DEV)
    for outs, *rest in got:
        assert all(torch.equal(a, b) for a, b in zip(rest, ref[1:]))
        assert all(torch.equal(a, b) for x, y in zip(outs, ref[0]) for a, b in zip(x, y))


def test_training_steps_on_changing_inputs():
    """Steps without a wait on inputs that change in place, against the same
    steps with a wait after each (Delta reads O and dO before the pass in front
    of it is complete)."""
    w = wl.Workload("pdl", wl.pack(DIALOGUES), 4, 2, 64, "bf16", 0.125, 1.0, 33)
    segs = ism.Segments.from_workload(w.segs, DEV)
    xs = [[(t.float() * f).bfloat16().to(DEV) for t in wl.attention_tensors(w)] for f in (1.0, 0.5, -1.5, 2.0)]
    live = [torch.empty_like(t) for t in xs[0]]
    o, lse = torch.empty_like(live[0]), torch.empty((4, live[0].shape[0]), device=DEV)

    def steps(waits):
        outs = []
        for i in range(12):
            for a, b in zip(live, xs[i % 4]):
                torch.mul(b, 1.0, out=a)
            ism.fwd(segs, *live[:3], w.softmax_scale, out=o, lse=lse)
            outs.append((o.clone(), *ism.bwd(segs, *live[:3], o, lse, live[3], w.softmax_scale)))
            if waits:
                torch.cuda.synchronize()
        torch.cuda.synchronize()
        return outs

    ref = steps(True)
    for _ in range(3):
        assert all(torch.equal(a, b) for x, y in zip(steps(False), ref) for a, b in zip(x, y))
    ism.check_status(DEV)
