"""The paired forward on the work counter against the static walk's results
(bit for bit: only which CTA takes a unit differs) and the oracle: fewer units
than CTAs, several a CTA, many single-tile dialogues (units whose second half is
empty), plans used again and again (planned forwards walk statically and leave
the plan as it is, so they may overlap), and the counter's place in every
workspace.
"""
import numpy as np
import pytest
import torch

from oracle import ism_oracle as orc
from paper_2408_00539_gb300 import ism
from paper_2408_00539_gb300 import workloads as wl

pytestmark = pytest.mark.gpu
DEV = "cuda:0"

SHORT = [([n], [n & 1]) for n in (1, 7, 127, 128, 100, 31)]
RAGGED = [([70, 150, 170, 300, 900], [0, 1, 0, 1, 0]), ([129], [0]), ([60, 257], [1, 0]), ([128], [1])]


@pytest.mark.parametrize("dialogues", [SHORT, RAGGED, SHORT * 40, RAGGED * 12], ids=["short", "ragged", "many_short",
                                                                                     "many_ragged"])
@pytest.mark.parametrize("hq,hkv,d", [(8, 2, 128), (3, 3, 128), (6, 2, 64), (4, 2, 64)])
def test_plan_and_plain_calls(dialogues, hq, hkv, d):
    w = wl.Workload("dyn", wl.pack(dialogues), hq, hkv, d, "bf16", d ** -0.5, 1.0, 21)
    q, k, v = wl.attention_tensors(w, with_dout=False)
    segs = ism.Segments.from_workload(w.segs, DEV)
    dev = [t.to(DEV) for t in (q, k, v)]
    o, lse = ism.fwd(segs, *dev, w.softmax_scale)
    plan = ism.Plan(segs, hq, hkv, d, torch.bfloat16, DEV)
    for _ in range(3):
        o2, lse2 = ism.fwd(segs, *dev, w.softmax_scale, plan=plan)
        assert torch.equal(o, o2) and torch.equal(lse, lse2)
    ism.check_status(DEV)
    if len(dialogues) < 10:
        ref = orc.attn_fwd(q, k, v, w.segs, w.softmax_scale)[0]
        err = np.abs(o.double().cpu().numpy() - ref)
        assert err.max() <= 2e-2 and err.mean() <= 2e-3


def test_head_pairs_match_the_static_walk():
    """The same dialogues few (counter) and many times over (static walk)."""
    w = wl.Workload("dyn", wl.pack(RAGGED), 32, 8, 128, "bf16", 128 ** -0.5, 1.0, 22)
    x = [t.to(DEV) for t in wl.attention_tensors(w, with_dout=False)]
    copies = 8  # 14 query tiles, 16 head pairs: 224 units, then 1792 (over eight a CTA)
    few = ism.fwd(ism.Segments.from_workload(w.segs, DEV), *x, w.softmax_scale)
    many_segs = ism.Segments.from_workload(wl.pack(RAGGED * copies), DEV)
    many = ism.fwd(many_segs, *(t.repeat(copies, 1, 1) for t in x), w.softmax_scale)
    ism.check_status(DEV)
    T = w.total_tokens
    for i in range(copies):
        assert torch.equal(many[0][i * T:(i + 1) * T], few[0])
        assert torch.equal(many[1][:, i * T:(i + 1) * T], few[1])


@pytest.mark.parametrize("hq,hkv,d", [(8, 2, 128), (3, 3, 128), (6, 2, 64)])
@pytest.mark.parametrize("rope", [False, True])
def test_planned_forwards_leave_the_plan_alone(hq, hkv, d, rope):
    """Forwards on one plan from two streams at once: the plan's bytes stay what
    the build wrote, and every result is the plain call's."""
    w = wl.Workload("dyn", wl.pack(RAGGED * 6), hq, hkv, d, "bf16", d ** -0.5, 1.0, 23)
    x = [t.to(DEV) for t in wl.attention_tensors(w, with_dout=False)]
    segs = ism.Segments.from_workload(w.segs, DEV)
    tables = tuple(torch.from_numpy(t).to(DEV) for t in wl.rope_tables(900, d)) if rope else ()
    call = ism.fwd_rope if rope else ism.fwd
    ref = call(segs, *x, *tables, w.softmax_scale)
    plan = ism.Plan(segs, hq, hkv, d, torch.bfloat16, DEV)
    torch.cuda.synchronize()
    before = plan.buffer.clone()
    streams = [torch.cuda.Stream(DEV) for _ in range(2)]
    torch.cuda.synchronize()
    outs = []
    for _ in range(20):
        for s in streams:
            with torch.cuda.stream(s):
                outs.append(call(segs, *x, *tables, w.softmax_scale, plan=plan))
    torch.cuda.synchronize()
    ism.check_status(DEV)
    assert torch.equal(plan.buffer, before)
    for out in outs:
        assert all(torch.equal(a, b) for a, b in zip(out, ref))
