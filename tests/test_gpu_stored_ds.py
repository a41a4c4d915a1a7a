"""dK/dV and dQ where the backward stores dS tiles: last query tiles of every
kind (their absent queries are neither stored nor contracted)."""
import numpy as np
import pytest
import torch

from oracle import ism_oracle as orc
from paper_2408_00539_gb300 import ism
from paper_2408_00539_gb300 import workloads as wl

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
TAILS = [([n], [1]) for n in (1, 8, 9, 64, 65, 120, 121, 128, 129, 136, 192, 193, 256)]


def _step(segs, x, scale):
    o, lse = ism.fwd(segs, *x[:3], scale)
    return ism.bwd(segs, *x[:3], o, lse, x[3], scale)


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
