"""dK/dV and dQ where the backward stores dS tiles: last query tiles of every
kind (their absent queries are neither stored nor contracted), and dQ with two
heads a unit against one (bit for bit: the same sums in the same order, only
shared loads)."""
import numpy as np
import pytest
import torch

from oracle import ism_oracle as orc
from paper_2408_00539_gb300 import ism
from paper_2408_00539_gb300 import workloads as wl

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
TAILS = [([n], [1]) for n in (1, 8, 9, 64, 65, 120, 121, 128, 129, 136, 192, 193, 256)]
RAGGED = [([70, 150, 170, 300], [0, 1, 0, 1]), ([129], [0]), ([60, 257], [1, 0]), ([128], [1])]


def _step(segs, x, scale, rope=None):
    if rope is None:
        o, lse = ism.fwd(segs, *x[:3], scale)
        return ism.bwd(segs, *x[:3], o, lse, x[3], scale)
    o, lse, q, k = ism.fwd_rope(segs, *x[:3], *rope, scale)
    return ism.bwd_rope(segs, q, k, x[2], o, lse, x[3], *rope, scale)


@pytest.mark.parametrize("hq,hkv,d", [(2, 2, 128), (4, 1, 128), (2, 1, 64)])
def test_last_tiles(hq, hkv, d):
    w = wl.Workload("tails", wl.pack(TAILS), hq, hkv, d, "bf16", d ** -0.5, 1.0, 41)
    host = wl.attention_tensors(w)
    got = _step(ism.Segments.from_workload(w.segs, DEV), [t.to(DEV) for t in host], w.softmax_scale)
    ism.check_status(DEV)
    ref = orc.attn_bwd(*host[:3], host[3], w.segs, w.softmax_scale)
    for a, b in zip(got, ref):
        # the repository's bf16 gradient bounds, and the results' own rounding
        # (2^-9 of a value) where single-token dialogues sum four heads' dO
        err = np.abs(a.double().cpu().numpy() - b)
        assert np.isfinite(err).all() and (err <= 2e-2 + 2.0 ** -9 * np.abs(b)).all() and err.mean() <= 4e-3


@pytest.mark.parametrize("hq,hkv", [(8, 4), (16, 4), (12, 2), (6, 2)])
@pytest.mark.parametrize("rope", [None, 32, 16])
def test_head_units(hq, hkv, rope):
    """Few copies of the dialogues (one head a unit) and many (two, where the KV
    heads have an even number); rotary tables aligned to 32 and to 16 bytes."""
    w = wl.Workload("units", wl.pack(RAGGED), hq, hkv, 128, "bf16", 128 ** -0.5, 1.0, 42)
    x = [t.to(DEV) for t in wl.attention_tensors(w)]
    tables = None
    if rope:
        tables = []
        for t in wl.rope_tables(800, 128):
            room = torch.zeros(t.size + 4, device=DEV)
            room[4 if rope == 16 else 0:][:t.size] = torch.from_numpy(t).to(DEV).flatten()
            tables.append(room[4 if rope == 16 else 0:][:t.size].view(t.shape))
    few = _step(ism.Segments.from_workload(w.segs, DEV), x, w.softmax_scale, tables)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    copies = sms * 10 // (12 * hq) + 2  # 12 query tiles a copy: above ten items an SM
    many = _step(ism.Segments.from_workload(wl.pack(RAGGED * copies), DEV), [t.repeat(copies, 1, 1) for t in x],
                 w.softmax_scale, tables)
    ism.check_status(DEV)
    T = w.total_tokens
    for a, b in zip(few, many):
        for i in range(copies):
            assert torch.equal(b[i * T:(i + 1) * T], a)
