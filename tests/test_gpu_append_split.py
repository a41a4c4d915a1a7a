"""Key-range split of the append forward: every number of parts the rule takes
(head pairs, query-tile pairs of odd groups, paged, head_dim 64), the halves of
e4m3, parts without key tiles, workspaces of the required size only, and the cache lengths
after each call.  Reference: the same call unsplit (ISM_PREFILL_SPLIT=0).

Tolerance, in the 2-norm against the whole item's result: at head_dim 128 P is
rounded to bf16 relative to a part's own maximum, so each of the two results is
off the exact one by up to 2^-9 for P (independent roundings of the terms of a
sum of zero-mean V) and 2^-9 for the output: 4 * 2^-9 between them.  At 64 P
keeps 16 bits, and only the output roundings differ, where the two sums fall on
either side of a boundary: 2^-9.  e4m3 P: 2^-4 in the place of 2^-9, uniform
roundings of zero mean: 4e-2.
"""
import ctypes as C

import numpy as np
import pytest
import torch

from oracle import ism_oracle as orc
from paper_2408_00539_gb300 import ism
from paper_2408_00539_gb300 import workloads as wl

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _inputs(hq, hkv, d, lens, ln, seed=3):
    gen = torch.Generator().manual_seed(seed)
    B, cap = len(lens), int(max(lens)) + ln + 3
    x = [torch.randn((B, ln, h, d), generator=gen).bfloat16() for h in (hq, hkv, hkv)]
    return x + [torch.randn((B, cap, hkv, d), generator=gen).bfloat16() for _ in range(2)]


def _call(monkeypatch, split, x, lens, ends, types, scale, workspace=None):
    lens = np.asarray(lens, np.int32)
    dev = [t.to(DEV) for t in x]
    cl = torch.from_numpy(lens.copy()).to(DEV)
    if split is not None:
        monkeypatch.setenv("ISM_PREFILL_SPLIT", str(split))
    ism.load().ism_debug_reload_env()
    try:
        o, lse = ism.prefill_append(*dev, cl, lens, ends, types, scale, workspace=workspace)
        ism.check_status(DEV)
    finally:
        monkeypatch.delenv("ISM_PREFILL_SPLIT", raising=False)
        ism.load().ism_debug_reload_env()
    assert np.array_equal(cl.cpu().numpy(), lens + x[0].shape[1])
    return o, lse, dev[3], dev[4]


def _same(got, ref, rel=2.0 ** -7):
    for a, b in zip(got[2:], ref[2:]):
        assert torch.equal(a, b)
    a, b = got[0].double(), ref[0].double()
    assert torch.isfinite(a).all() and float((a - b).norm() / b.norm()) <= rel
    assert float((got[1] - ref[1]).abs().max()) <= 2e-5


# short and long caches, one or several query tiles, ragged lengths, one key tile (no split)
@pytest.mark.parametrize("lens,ln", [([3000], 40), ([5], 7), ([900, 1, 300], 130), ([2500, 4096], 300), ([130], 128)])
@pytest.mark.parametrize("hq,hkv,d", [(8, 2, 128), (4, 4, 128), (6, 2, 64), (4, 2, 64), (3, 1, 128)])
def test_split_matches_whole(monkeypatch, hq, hkv, d, lens, ln):
    x = _inputs(hq, hkv, d, lens, ln)
    ends, types = [ln // 2, ln], [0, 1]
    whole = _call(monkeypatch, 0, x, lens, ends, types, d ** -0.5)
    got = _call(monkeypatch, None, x, lens, ends, types, d ** -0.5)
    _same(got, whole, 2.0 ** (-9 if d == 64 else -7))
    # against the oracle, sequence 0
    c = lens[0]
    segs = wl.pack([([c] + [c + e for e in ends], [1] + types)])
    full = [torch.cat([h[0, :c], n[0]]) for h, n in ((x[3], x[1]), (x[4], x[2]))]
    q = torch.cat([torch.zeros((c, hq, d), dtype=torch.bfloat16), x[0][0]])
    if c <= 3000 and ln <= 130:
        ref = orc.attn_fwd(q, *full, segs, d ** -0.5)[0][c:]
        err = np.linalg.norm(got[0][0].double().cpu().numpy() - ref) / np.linalg.norm(ref)
        assert err <= (2.0 ** -9 + 2.0 ** -14 if d == 64 else 4e-3)


def test_required_workspace_only(monkeypatch):
    """The workspace reported before the split took more parts is still enough
    (fewer parts), a smaller one is refused."""
    x = _inputs(8, 2, 128, [3000], 100)
    B, ln, hq, d = x[0].shape
    items = B * 1 * hq // 2
    head = sum((n + 255) // 256 * 256 for n in (4 * B, 4 * B * ln, 32 * B, 4 * B, 4 * B))
    need = head + items * 4 * 128 * 128 * 4 + items * 4 * 128 * 2 * 4 + 256
    ws = ism._workspace(need, DEV)
    whole = _call(monkeypatch, 0, x, [3000], [ln], [0], d ** -0.5)
    _same(_call(monkeypatch, None, x, [3000], [ln], [0], d ** -0.5, workspace=ws), whole)
    assert ism.append_workspace_size(x[0], x[1], d ** -0.5) > need
    lib = ism.load()
    dev = [t.to(DEV) for t in x]
    ch, se, st = np.array([3000], np.int32), np.array([ln], np.int32), np.array([0], np.uint8)
    sh = ism._shape(x[0], x[1], d ** -0.5)
    o = torch.empty_like(dev[0])
    code = lib.ism_attn_prefill_append(
        C.byref(sh), B, *(ism._ptr(t) for t in dev[:3]), ln, se.ctypes.data, st.ctypes.data, 1, ism._ptr(dev[3]),
        ism._ptr(dev[4]), x[3].shape[1], ism._ptr(torch.tensor([3000], dtype=torch.int32, device=DEV)), ch.ctypes.data,
        ism._ptr(o), None, ism._ptr(ws), need - 256, None)
    assert code == 5


@pytest.mark.parametrize("hq,hkv", [(8, 2), (3, 3)])
def test_split_e4m3_and_paged(monkeypatch, hq, hkv):
    lens, ln, d = np.array([1500, 700], np.int32), 60, 128
    x = _inputs(hq, hkv, d, lens, ln)
    out = []
    for split in ("0", None):
        if split:
            monkeypatch.setenv("ISM_PREFILL_SPLIT", split)
        else:
            monkeypatch.delenv("ISM_PREFILL_SPLIT", raising=False)
        ism.load().ism_debug_reload_env()
        e8 = [(t.float() / 0.01).clamp(-448, 448).to(torch.float8_e4m3fn).to(DEV) for t in x]
        cl = torch.from_numpy(lens.copy()).to(DEV)
        o8, l8 = ism.prefill_append_e4m3(*e8, cl, lens, [ln], [0], 0.01, 0.01, 0.01, d ** -0.5)
        # pages of 128 in reverse order
        pages = [-(-(int(c) + ln) // 128) for c in lens]
        table = np.zeros((2, max(pages)), np.int32)
        ids = np.arange(sum(pages))[::-1]
        table[0, :pages[0]], table[1, :pages[1]] = ids[:pages[0]], ids[pages[0]:]
        pool = [torch.zeros((sum(pages) * 128, hkv, d), dtype=torch.bfloat16) for _ in range(2)]
        for b, c in enumerate(lens):
            for p in range(int(c)):
                for i in range(2):
                    pool[i][table[b, p // 128] * 128 + p % 128] = x[3 + i][b, p]
        pool = [t.to(DEV) for t in pool]
        cl2 = torch.from_numpy(lens.copy()).to(DEV)
        op, lp = ism.prefill_append_paged(*(t.to(DEV) for t in x[:3]), *pool, 128, torch.from_numpy(table).to(DEV),
                                          table, cl2, lens, [ln], [0], d ** -0.5)
        ism.check_status(DEV)
        out.append((o8, l8, op, lp, *pool))
    ism.load().ism_debug_reload_env()
    a, b = out
    assert float((a[0].double() - b[0].double()).norm() / a[0].double().norm()) <= 4e-2
    _same((b[2], b[3], b[4], b[5]), (a[2], a[3], a[4], a[5]))
    contiguous = _call(monkeypatch, None, x, lens, [ln], [0], d ** -0.5)
    assert torch.equal(contiguous[0], b[2]) and torch.equal(contiguous[1], b[3])


@pytest.mark.parametrize("hq,hkv,batch,cached,split", [(8, 2, 2, 1500, "8"), (3, 3, 2, 1500, "6"), (32, 8, 10, 8200, None)])
def test_e4m3_halves(monkeypatch, hq, hkv, batch, cached, split):
    """e4m3 in two halves of the key range, forced on all items (an even and an
    odd group) and by its own rule (items past a whole round, long caches).  Both
    results are off the exact one by their roundings of P, and differ from each
    other: the split was taken."""
    ln, d, f = 60, 128, 0.01
    gen = torch.Generator(device=DEV).manual_seed(4)

    def e8(*shape):
        x = torch.randn(shape, generator=gen, device=DEV, dtype=torch.bfloat16)
        return (x.float() / f).clamp(-448, 448).to(torch.float8_e4m3fn)

    x = [e8(batch, ln, h, d) for h in (hq, hkv, hkv)] + [e8(batch, cached + ln, hkv, d) for _ in range(2)]
    lens = np.full((batch,), cached, np.int32)
    out = []
    for n in ("0", split):
        if n is None:
            monkeypatch.delenv("ISM_PREFILL_SPLIT", raising=False)
        else:
            monkeypatch.setenv("ISM_PREFILL_SPLIT", n)
        ism.load().ism_debug_reload_env()
        try:
            out.append(ism.prefill_append_e4m3(*x, torch.from_numpy(lens.copy()).to(DEV), lens, [ln], [0], f, f, f,
                                               d ** -0.5))
            ism.check_status(DEV)
        finally:
            monkeypatch.delenv("ISM_PREFILL_SPLIT", raising=False)
            ism.load().ism_debug_reload_env()
    whole, got = (o.double() for o, _ in out)
    assert torch.isfinite(got).all() and not torch.equal(whole, got)
    assert float((whole - got).norm() / whole.norm()) <= 4e-2
    assert float((out[0][1] - out[1][1]).abs().max()) <= 2e-5
    # the last sequence against 64 bits (the rule splits the last items)
    kv = [(torch.cat([c[-1, :cached], n[-1]]).double() * f) for c, n in ((x[3], x[1]), (x[4], x[2]))]
    q = x[0][-1].double() * f
    for h in range(0, hq, max(1, hq // 4)):
        k, v = (t[:, h // (hq // hkv)] for t in kv)
        exact = torch.softmax(q[:, h] @ k.T * d ** -0.5, dim=1) @ v
        assert float((got[-1, :, h] - exact).norm() / exact.norm()) <= 4e-2
