"""Single-token steps of the bf16 tensor-core decode, whose CTAs share out the
tiles of all caches: ragged and equal lengths, more sequences than a warp scans
at once, shares of one tile and of several items, caches at tile edges, and few
long caches (each starting at a CTA's share).  Reference: the CUDA-core decode
of the same step (ISM_DECODE_NO_TC=1, fp32 P) and the oracle for one of them.

Tolerance: in equal chunks P is rounded to bf16 for P V (2^-9 of independent
terms) and the output to bf16 (2^-9), the reference rounds its output (2^-9):
3 * 2^-9 in the 2-norm; LSE 2^-9, as its sum is of the rounded P (each term off by
at most 2^-9).  The row split keeps P to 16 bits.
"""
import numpy as np
import pytest
import torch

from paper_2408_00539_gb300 import ism

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
RNG = np.random.default_rng(5)

CASES = {
    "one": [0], "one_long": [3001], "edges": [126, 127, 128, 255, 256],
    "ragged": [int(x) for x in RNG.integers(1, 4000, 40)],
    "many_short": [int(x) for x in RNG.integers(0, 300, 300)],
    "many_equal": [200] * 130, "equal_long": [9000] * 3, "one_among": [20000] + [3] * 20,
}


def _step(monkeypatch, no_tc, lens, q, k, v, kc, vc):
    if no_tc:
        monkeypatch.setenv("ISM_DECODE_NO_TC", "1")
    ism.load().ism_debug_reload_env()
    try:
        kc, vc = kc.clone(), vc.clone()
        lens = np.asarray(lens, np.int32)
        cl = torch.from_numpy(lens.copy()).to(DEV)
        o, lse = ism.prefill_append(q, k, v, kc, vc, cl, lens, [1], [1], 128 ** -0.5)
        ism.check_status(DEV)
    finally:
        monkeypatch.delenv("ISM_DECODE_NO_TC", raising=False)
        ism.load().ism_debug_reload_env()
    assert np.array_equal(cl.cpu().numpy(), lens + 1)
    return o, lse


def _compare(monkeypatch, lens, hq, hkv):
    gen = torch.Generator(device=DEV).manual_seed(len(lens))
    B, cap = len(lens), max(lens) + 1
    q, k, v = (torch.randn((B, 1, h, 128), generator=gen, device=DEV).bfloat16() for h in (hq, hkv, hkv))
    kc, vc = (torch.randn((B, cap, hkv, 128), generator=gen, device=DEV).bfloat16() for _ in range(2))
    got, ref = (_step(monkeypatch, no_tc, lens, q, k, v, kc, vc) for no_tc in (False, True))
    a, b = got[0].double(), ref[0].double()
    assert torch.isfinite(a).all() and float((a - b).norm() / b.norm()) <= 3 * 2.0 ** -9
    assert float((got[1] - ref[1]).abs().max()) <= 2.0 ** -9
    # per sequence too: a part lost or taken twice in a short one would hide in the whole
    err = (a - b).flatten(1).norm(dim=1) / b.flatten(1).norm(dim=1)
    assert float(err.max()) <= 6 * 2.0 ** -9


@pytest.mark.parametrize("name", sorted(CASES))
@pytest.mark.parametrize("hq,hkv", [(8, 2), (6, 6), (32, 4)])
def test_matches_cuda_cores(monkeypatch, name, hq, hkv):
    _compare(monkeypatch, CASES[name], hq, hkv)


@pytest.mark.parametrize("name", ["edges", "ragged", "one_among"])
@pytest.mark.parametrize("hq,hkv", [(3, 3), (16, 16), (24, 12)])
def test_head_lanes(monkeypatch, name, hq, hkv):
    """One, eight (two groups in the row) and four neighbouring heads a share."""
    _compare(monkeypatch, CASES[name], hq, hkv)


@pytest.mark.parametrize("lens,hkv", [([150000], 1), ([195000], 2), ([190000, 5], 1)])
def test_long_caches(monkeypatch, lens, hkv):
    """Few caches of more than 62 shares: each starts at a share of its own."""
    _compare(monkeypatch, lens, 4 * hkv, hkv)


@pytest.mark.parametrize("page", [128, 256])
def test_paged_matches_contiguous(page):
    lens = np.array([500, 1, 127, 900], np.int32)
    gen = torch.Generator().manual_seed(9)
    B, hq, hkv = 4, 8, 2
    q, k, v = (torch.randn((B, 1, h, 128), generator=gen).bfloat16() for h in (hq, hkv, hkv))
    kc, vc = (torch.randn((B, 1024, hkv, 128), generator=gen).bfloat16() for _ in range(2))
    per = 1024 // page
    table = np.random.default_rng(1).permutation(B * per).astype(np.int32).reshape(B, per)
    pools = []
    for c in (kc, vc):
        pool = torch.empty((B * per, page, hkv, 128), dtype=torch.bfloat16)
        pool[torch.from_numpy(table.reshape(-1).astype(np.int64))] = c.reshape(B * per, page, hkv, 128)
        pools.append(pool.reshape(-1, hkv, 128).to(DEV))
    new = [t.to(DEV) for t in (q, k, v)]
    a = ism.prefill_append(*new, kc.to(DEV), vc.to(DEV), torch.from_numpy(lens.copy()).to(DEV), lens, [1], [1], 0.09)
    b = ism.prefill_append_paged(*new, *pools, page, torch.from_numpy(table).to(DEV), table,
                                 torch.from_numpy(lens.copy()).to(DEV), lens, [1], [1], 0.09)
    ism.check_status(DEV)
    assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1])


@pytest.mark.parametrize("hq,hkv", [(8, 2), (16, 2), (32, 2)])
@pytest.mark.parametrize("value", [None, "inf", "nan"])
def test_values_to_16_bits(monkeypatch, hq, hkv, value):
    """The row split keeps P to 16 bits: against the CUDA-core decode (fp32 P)
    only output roundings differ where the two sums fall on either side of a
    boundary, so the 2-norm of the difference stays far below one rounding
    (2^-12; a bf16 P gives 1.5e-3).  An Inf or NaN among the values comes out
    as there."""
    lens = [700, 3000, 130, 1900]
    gen = torch.Generator(device=DEV).manual_seed(11)
    q, k, v = (torch.randn((4, 1, h, 128), generator=gen, device=DEV).bfloat16() for h in (hq, hkv, hkv))
    kc, vc = (torch.randn((4, 3001, hkv, 128), generator=gen, device=DEV).bfloat16() for _ in range(2))
    if value:
        vc[1, 1500, 0, 7] = vc[3, 40, 1, 100] = float(value)
    got, ref = (_step(monkeypatch, no_tc, lens, q, k, v, kc, vc) for no_tc in (False, True))
    a, b = got[0].double(), ref[0].double()
    ok = torch.isfinite(b)
    assert torch.equal(torch.isnan(a), torch.isnan(b)) and torch.equal(torch.isinf(a), torch.isinf(b))
    assert int((~ok).sum()) == (2 * (hq // hkv) if value else 0)
    assert float((a - b)[ok].norm() / b[ok].norm()) <= 2.0 ** -12
    assert float((got[1] - ref[1]).abs().max()) <= 1e-5


@pytest.mark.parametrize("name", ["one_long", "ragged", "many_short", "edges"])
@pytest.mark.parametrize("off", [-1000, -130, -1, 500])
def test_host_lengths_that_lag(name, off):
    """Lengths on the device that the host's copy does not know (a captured step
    replayed): the keys past what the launch was laid out for go to the last
    share, in place of being left out; a copy ahead of the device leaves shares
    without keys.  Reference: the same step with the right copy, which shares
    the tiles out otherwise (output roundings on either side of a boundary)."""
    lens = np.array(CASES[name], np.int32)
    gen = torch.Generator(device=DEV).manual_seed(3)
    B, cap, hq, hkv = len(lens), int(lens.max()) + 600, 8, 2
    x = [torch.randn((B, 1, h, 128), generator=gen, device=DEV).bfloat16() for h in (hq, hkv, hkv)]
    caches = [torch.randn((B, cap, hkv, 128), generator=gen, device=DEV).bfloat16() for _ in range(2)]
    out = []
    for host in (lens, np.maximum(lens + off, 0)):
        cl = torch.from_numpy(lens.copy()).to(DEV)
        out.append(ism.prefill_append(*x, *(c.clone() for c in caches), cl, host, [1], [1], 128 ** -0.5))
        ism.check_status(DEV)
        assert np.array_equal(cl.cpu().numpy(), lens + 1)
    a, b = out[1][0].double(), out[0][0].double()
    err = (a - b).flatten(1).norm(dim=1) / b.flatten(1).norm(dim=1)
    assert torch.isfinite(a).all() and float(err.max()) <= 2.0 ** -9
    assert float((a - b).norm() / b.norm()) <= 2.0 ** -12
    assert float((out[1][1] - out[0][1]).abs().max()) <= 1e-5
